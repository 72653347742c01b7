// mm_clip.cuh -- arithmetic shared by the clipping kernels: the FP64 plane
// intersection and plane test every decision rests on, and the FP32 ones with
// their error bounds.
#pragma once

#include "mm_fp64.cuh"
#include "mm_internal.cuh"

namespace mm {

constexpr unsigned FULL = 0xffffffffu;
// Rarely taken integer work of the gather, kept out of line so that the hot
// loop around it stays small (the kernel is sensitive to instruction-cache
// misses): floor(a / b) for b > 0 (images beyond the neighbouring boxes), and
// the bin offsets of entry t of ring block rh of side nb = 2 rh + 1 (rings 3
// and beyond).
static __device__ __noinline__ int floordiv(int a, int b) { return a >= 0 ? a / b : -((-a + b - 1) / b); }
static __device__ __noinline__ int3 ring_offset(int t, int nb, int rh)
{
    return make_int3(t % nb - rh, (t / nb) % nb - rh, t / (nb * nb) - rh);
}

__device__ __forceinline__ unsigned lanemask_lt() { return (1u << (threadIdx.x & 31)) - 1u; }

// Magnitude order of doubles by their bit patterns (non-negative values, or
// absolute values): an integer comparison in place of an FP64 one.
__device__ __forceinline__ long long abs_bits(double x)
{
    return __double_as_longlong(x) & 0x7fffffffffffffffLL;
}
// Intersection of planes a, b, c in FP64 with explicitly rounded operations
// (so every caller gets the same bits):
// x = (o_a (q_b x q_c) + q_a x (o_c q_b - o_b q_c)) / det(q_a, q_b, q_c),
// 30 FP64 operations (Cramer's rule with all three cross products: 36).
__device__ __forceinline__ void solve64(double ax, double ay, double az, double ao, double bx, double by, double bz,
                                        double bo, double cx, double cy, double cz, double co, double &x, double &y,
                                        double &z)
{
    const double nx = __fma_rn(by, cz, -__dmul_rn(bz, cy)), ny = __fma_rn(bz, cx, -__dmul_rn(bx, cz)),
                 nz = __fma_rn(bx, cy, -__dmul_rn(by, cx));
    const double dx = __fma_rn(co, bx, -__dmul_rn(bo, cx)), dy = __fma_rn(co, by, -__dmul_rn(bo, cy)),
                 dz = __fma_rn(co, bz, -__dmul_rn(bo, cz));
    const double inv = rcp64(__fma_rn(ax, nx, __fma_rn(ay, ny, __dmul_rn(az, nz))));
    x = __dmul_rn(__fma_rn(ao, nx, __fma_rn(ay, dz, -__dmul_rn(az, dy))), inv);
    y = __dmul_rn(__fma_rn(ao, ny, __fma_rn(az, dx, -__dmul_rn(ax, dz))), inv);
    z = __dmul_rn(__fma_rn(ao, nz, __fma_rn(ax, dy, -__dmul_rn(ay, dx))), inv);
}
template <class S_t>
__device__ __forceinline__ void vertex64(const S_t &S, int a, int b, int c, double &x, double &y, double &z)
{
    solve64(S.px[a], S.py[a], S.pz[a], S.po[a], S.px[b], S.py[b], S.pz[b], S.po[b], S.px[c], S.py[c], S.pz[c], S.po[c],
            x, y, z);
}

// The exact-path predicate: is vertex v strictly beyond the plane x.q <= off?
__device__ __forceinline__ bool beyond64(double qx, double qy, double qz, double off, double x, double y, double z)
{
    return __fma_rn(qx, x, __fma_rn(qy, y, __dmul_rn(qz, z))) > off;
}

// |q|^2 / 2 from the bit pattern of |q|^2: halving a normal double lowers its
// exponent by one, an integer operation.
__device__ __forceinline__ double half_of(long long d2bits)
{
    if (((d2bits >> 52) & 0x7ff) > 1) return __longlong_as_double(d2bits - (1LL << 52));
    return 0.5 * __longlong_as_double(d2bits);
}

__device__ __forceinline__ long long r2_bits64(double x, double y, double z)
{
    return __double_as_longlong(__fma_rn(x, x, __fma_rn(y, y, __dmul_rn(z, z))));
}

// Square root within 2^-23 (the hardware's), for bounds
__device__ __forceinline__ float sqrt_fast(float x)
{
    float r;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// FP32 |q| of a plane with offset o = |q|^2 / 2, for the error bound below (the
// correctly rounded root costs the grouped clipper, which forms three of them a
// vertex, 1.5 %: 512 boxes 194.2 -> 197.7 ms)
__device__ __forceinline__ float plane_length(float o) { return sqrt_fast(2.0f * o); }

// Intersection of planes a, b, c in FP32 with a bound on its distance to the
// exact intersection.  With P = |q_a||q_b||q_c|, H = P / |det| >= 1 and
// u = 2^-24, first-order rounding analysis of Cramer's rule (inputs rounded
// to FP32, cross products, determinant, numerator, scaling) gives
// |v~ - v| <= u H (5.5 sum|q| + 13 |v|); the bound used is three times that,
// which covers the roundings of the bound itself (plane_length's, H's).
// Ill-conditioned intersections get an infinite bound (always checked in FP64).
// la, lb, lc are the planes' |q| (plane_length).  Products that feed a sum are
// written as such, so that every kernel gets the same bits.
__device__ __forceinline__ void solve32(const float4 Pa, const float4 Pb, const float4 Pc, float la, float lb, float lc,
                                        float &x, float &y, float &z, float &err)
{
    const float ax = Pa.x, ay = Pa.y, az = Pa.z, ao = Pa.w;
    const float bx = Pb.x, by = Pb.y, bz = Pb.z, bo = Pb.w;
    const float cx = Pc.x, cy = Pc.y, cz = Pc.z, co = Pc.w;
    const float bcx = fmaf(by, cz, -bz * cy), bcy = fmaf(bz, cx, -bx * cz), bcz = fmaf(bx, cy, -by * cx);
    const float cax = fmaf(cy, az, -cz * ay), cay = fmaf(cz, ax, -cx * az), caz = fmaf(cx, ay, -cy * ax);
    const float abx = fmaf(ay, bz, -az * by), aby = fmaf(az, bx, -ax * bz), abz = fmaf(ax, by, -ay * bx);
    const float det = fmaf(ax, bcx, fmaf(ay, bcy, az * bcz));
    const float inv = __frcp_rn(det);
    x = __fmul_rn(fmaf(ao, bcx, fmaf(bo, cax, co * abx)), inv);
    y = __fmul_rn(fmaf(ao, bcy, fmaf(bo, cay, co * aby)), inv);
    z = __fmul_rn(fmaf(ao, bcz, fmaf(bo, caz, co * abz)), inv);
    const float H = la * lb * lc * fabsf(inv);  // P / |det| through the reciprocal (the factor 3 covers its ulp)
    const float vn = fabsf(x) + fabsf(y) + fabsf(z);
    const float u = 5.9604645e-8f;
    err = __fmul_rn(3.0f * u * H, fmaf(5.5f, la + lb + lc, 13.0f * vn));
    // The analysis assumes no FP32 underflow or overflow: the numerators grow
    // like |q|^4 and the determinant like |q|^3, so planes much nearer than
    // 2^-28 or farther than 2^28 (tiny or huge boxes) are solved exactly.
    const float qlo = fminf(la, fminf(lb, lc)), qhi = fmaxf(la, fmaxf(lb, lc));
    if (!(u * H < 1e-3f) || !(err < 1e30f) || !(qlo >= 3.7252903e-9f) || !(qhi <= 268435456.0f))
        err = __int_as_float(0x7f800000);  // +inf
}
// An ill-conditioned intersection is solved in FP64; of its FP32 rounding the
// error is then one rounding per axis.
__device__ __forceinline__ void rounded_vertex(double X, double Y, double Z, float &x, float &y, float &z, float &err)
{
    x = (float)X;
    y = (float)Y;
    z = (float)Z;
    err = fmaf(1.2e-7f, fabsf(x) + fabsf(y) + fabsf(z), 1e-38f);
}
// FP32 bound of (|v| + err)^2 <= |v|^2 + err (2 |v|_1 + err), short of a factor
// that covers its roundings.
__device__ __forceinline__ float vertex_r2(float x, float y, float z, float err)
{
    const float l1 = fabsf(x) + fabsf(y) + fabsf(z);
    return fmaf(err, fmaf(2.0f, l1, err), fmaf(x, x, fmaf(y, y, __fmul_rn(z, z))));
}
template <class S_t>
__device__ __forceinline__ void vertex32(const S_t &S, int a, int b, int c, float &x, float &y, float &z,
                                         float &err)
{
    solve32(S.pf[a], S.pf[b], S.pf[c], S.pfn[a], S.pfn[b], S.pfn[c], x, y, z, err);
}

// Fan about a face polygon's first vertex v0 with offsets d = v - v0 formed
// once per vertex.  The offsets lie in the plane x.q = o, so d_a x d_b is
// parallel to q and q . (d_a x d_b) equals (|q|^2 / q_k) times the 2-D cross
// product of the two coordinates other than k, the axis where |q| is largest.
// Edge (a, b) spans the triangle (v0, a, b) with 2-D weight w; with W = sum w:
// area = |W| |q| / (2 |q_k|), pyramid volume A |q| / 6 = |W| |q|^2 / (12 |q_k|),
// centroid offset = sum w (d_a + d_b) / (3 W) in the two kept coordinates, and
// in the k-th from the plane equation q . offset = 0.  Offsets from v0 keep
// the rounding relative to the face's own size.
struct FaceFan {
    double au = 0.0, av = 0.0;  // offset of the current vertex
    double W = 0.0, su = 0.0, sv = 0.0;
    // the first edge from v0: a triangle of zero weight (edge() gives the same bits)
    __device__ __forceinline__ void begin(double bu, double bv)
    {
        au = bu;
        av = bv;
    }
    __device__ __forceinline__ void edge(double bu, double bv)
    {
        const double w = __fma_rn(au, bv, -__dmul_rn(av, bu));
        W = __dadd_rn(W, w);
        su = __fma_rn(w, __dadd_rn(au, bu), su);
        sv = __fma_rn(w, __dadd_rn(av, bv), sv);
        au = bu;
        av = bv;
    }
};
__device__ __forceinline__ int fan_axis(double qx, double qy, double qz)
{
    const long long aqx = abs_bits(qx), aqy = abs_bits(qy), aqz = abs_bits(qz);
    return (aqx >= aqy && aqx >= aqz) ? 0 : (aqy >= aqz ? 1 : 2);
}
// Area, centroid (first vertex at x0, y0, z0) and pyramid volume of the face
// in plane q, o whose fan F runs in the coordinates other than k.
__device__ __forceinline__ void face_of_fan(const FaceFan &F, int k, double qx, double qy, double qz, double o,
                                            double x0, double y0, double z0, double &area, double &fx, double &fy,
                                            double &fz, double &vp)
{
    const double qk = k == 0 ? qx : (k == 1 ? qy : qz);
    const double q1 = k == 0 ? qy : qx, q2 = k == 2 ? qy : qz;
    // 1 / q_k and 1 / (3 W) from one reciprocal of 3 W q_k; a face
    // of zero fan weight (area 0) takes 0 for both
    const double w3 = __dmul_rn(3.0, F.W);
    const bool nz = abs_bits(F.W) != 0;
    const double r = nz ? rcp64(__dmul_rn(w3, qk)) : 0.0;
    const double iq = __dmul_rn(w3, r);
    const double s = fabs(__dmul_rn(F.W, iq));            // |W / q_k|
    area = __dmul_rn(s, __dmul_rn(o, rsqrt64(2.0 * o)));  // o / |q| = |q| / 2
    vp = __dmul_rn(s, __dmul_rn(o, 1.0 / 6.0));           // |q|^2 / 12
    const double i3w = __dmul_rn(qk, r);
    const double du = __dmul_rn(F.su, i3w), dv = __dmul_rn(F.sv, i3w);
    const double dk = __dmul_rn(-__fma_rn(q1, du, __dmul_rn(q2, dv)), iq);
    fx = __dadd_rn(x0, k == 0 ? dk : du);
    fy = __dadd_rn(y0, k == 1 ? dk : (k == 0 ? du : dv));
    fz = __dadd_rn(z0, k == 2 ? dk : dv);
}

}  // namespace mm
