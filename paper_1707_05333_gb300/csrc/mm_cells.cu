// mm_cells.cu -- the filtered clipper for ordinary cells.
//
// The same cell construction as k_clip (mm_clip.cu), with the same decisions,
// the same plane order and the same FP64 geometry bit for bit, laid out for
// the usual cell of 10-30 faces.  Cells are clipped with G lanes each: 32/G
// cells share a warp, so the control, ballots and topology updates of one
// instruction stream serve 32/G cells, and a cut's handful of removed and new
// vertices fill the G lanes instead of a fraction of 32.  Then the warp forms
// the FP64 geometry of its cells together, with full lanes (warp_geometry).
//
// What bounds it and what it measured (GB300, jittered 64^3 lattice and
// 200003 random generators, ncu durations; k_clip took 5.89 and 8.89 ms):
// 2.6 and 4.2 ms, of dependent latencies with 15 warps an SM (3.4 KB of
// shared memory a cell, 128 registers): 1.6 instructions a cycle, 4920 a cell
// against k_clip's 14200, and the FP64 pipe 55 % busy with 108 instructions a
// cell against 236.  Random cells take 11600 instructions at 1.8 a cycle, with
// 19 active lanes for the lattice's 24: cells of unlike length share a warp.
// (18 warps an SM at 96 registers gained nothing: the misses of the
// instruction cache doubled.)
//  * Loops are kept rolled: unrolled, the body outgrew the instruction cache
//    and half of the cycles went to fetching it (5.3 and 13.0 ms).
//  * Screening candidates a lane each after the first SCREEN instead of trying
//    all one by one: random generators 4.33 -> 3.58 ms (clipping alone).
//  * The library's divisions, for the ends of the range only, stand out of line:
//    tessellation of a 128^3 lattice 24.5 -> 24.0 ms.  Unrolling the vertex loop
//    twice, or the plane-test loop four times, costs 11 and 4 % for the
//    instruction cache.
//  * The geometry as a kernel of its own (1.45 and 1.10 ms, FP64 pipe 84 %
//    busy, after 1.70 and 3.58 ms of clipping) left the FP64 pipe idle in one
//    kernel and the issue slots in the other: 3.15 and 4.68 ms in all, here
//    2.88 and 4.33 before the shorter FP64 sequences (mm_fp64.cuh, solve64).
//
// A cell that outgrows these lists (more than 32 live planes, 56 vertices, 32
// new vertices in a cut, CELL_RINGS search rings), holds a coincident
// generator or has an inconsistent cut goes to a list that the warp-per-cell
// clipper works through next, so nothing is refused here.
#include <cstddef>

#include "mm_clip.cuh"

namespace mm {

namespace {

constexpr int CPM = 32;    // live planes: one bit of a word
constexpr int CTM = 56;    // vertices
constexpr int CNS = 32;    // new (and removed) vertices of one cut
constexpr int CCB = 64;    // candidate buffer, flushed as in k_clip
constexpr int CELL_RINGS = 6;
constexpr int SCREEN = 8;     // candidates of a new cell tried unscreened (16: 2.7 % slower on lattices, 4: 4 %)
constexpr int LANES = 8;   // lanes a cell (16 lanes: jittered 64^3 2.35 ms for 1.70, random generators the same)
constexpr unsigned BOX_PLANE = 31u << 27;  // plane reference of box face k: BOX_PLANE | k
constexpr unsigned IDX_MASK = 0x7ffffffu;  // sorted index of a plane reference (MM_MAX_CELLS < 2^27)
static_assert(MM_MAX_CELLS < (1LL << 27), "a plane reference holds the index in 27 bits");

struct __align__(16) CellSmem {
    float4 tf[CTM];       // vertex and its error bound
    float4 pf[CPM];       // FP32 planes (q, o)
    float4 cf[CCB];       // FP32 candidates (q, |q|^2 / 2)
    unsigned cid[CCB];    // sorted index | image code << 27
    unsigned bin[32];     // the chunk's bins: first sorted index | generators << 27
    unsigned bm[CPM];     // removed directed edges
    unsigned pid[CPM];    // plane references: sorted index | image code << 27
    double off[9];        // image offsets s L - p: off[3 d + s + 1]
    float offf[9];
    unsigned short vtri[CTM]; // the vertices' triangles a | b << 5 | c << 10
    unsigned short tri[CNS];  // new triangles
    unsigned char hole[CNS];  // removed vertices
    unsigned char bcode[32];  // sx | sy << 2 | sz << 4 | self << 6 of the bins
    unsigned char perm[CCB];  // candidates in order
    int pad[5];
};
// eight blocks of two warps (eight cells each) an SM; the cells of a warp start in different banks
static_assert(sizeof(CellSmem) % 32 == 16 && 8 * (8 * sizeof(CellSmem) + 1024) <= 228 * 1024, "shared memory of a cell");

// Bins of the search shells r = 1 (with the home bin) .. CELL_RINGS in k_clip's order and
// chunks of 32 of the (2r+1)^3 block: offsets + 8 as x | y << 4 | z << 8, and
// where each chunk starts.
struct Shells {
    unsigned short bin[13 * 13 * 13];
    unsigned short chunk[160];  // first entry of chunk c (all shells' chunks in a row)
    unsigned char first[CELL_RINGS + 2];  // first chunk of shell r
};
constexpr Shells make_shells()
{
    Shells t{};
    int nb = 0, nc = 0;
    for (int r = 1; r <= CELL_RINGS; ++r) {
        t.first[r] = (unsigned char)nc;
        const int s = 2 * r + 1, total = s * s * s;
        for (int i = 0; i < total; ++i) {
            if (i % 32 == 0) t.chunk[nc++] = (unsigned short)nb;
            const int x = i % s - r, y = (i / s) % s - r, z = i / (s * s) - r;
            const int ax = x < 0 ? -x : x, ay = y < 0 ? -y : y, az = z < 0 ? -z : z;
            const int ch = ax > ay ? (ax > az ? ax : az) : (ay > az ? ay : az);
            if (r == 1 || ch == r) t.bin[nb++] = (unsigned short)((x + 8) | (y + 8) << 4 | (z + 8) << 8);
        }
    }
    t.first[CELL_RINGS + 1] = (unsigned char)nc;
    t.chunk[nc] = (unsigned short)nb;
    return t;
}
__device__ const Shells SHELLS = make_shells();

// FP64 plane of a reference: q = r_j + s L - p and o = |q|^2 / 2.
__device__ __forceinline__ void plane64(const double *off, unsigned ref, const double4_32a *__restrict__ sorted,
                                        const BoxDev *gp, double &qx, double &qy, double &qz, double &o)
{
    const unsigned code = ref >> 27;
    if (code == 31u) {
        const int k = (int)(ref & 7u), d = k >> 1;
        const double L = gp->L[d], sL = (k & 1) ? -L : L;
        qx = d == 0 ? sL : 0.0;
        qy = d == 1 ? sL : 0.0;
        qz = d == 2 ? sL : 0.0;
        o = half_of(__double_as_longlong(__dmul_rn(L, L)));
        return;
    }
    const double4_32a P = sorted[ref & IDX_MASK];
    const unsigned dz = code / 9u, r = code - 9u * dz, dy = r / 3u, dx = r - 3u * dy;
    qx = __dadd_rn(P.x, off[dx]);
    qy = __dadd_rn(P.y, off[3 + dy]);
    qz = __dadd_rn(P.z, off[6 + dz]);
    o = half_of(__double_as_longlong(__fma_rn(qx, qx, __fma_rn(qy, qy, __dmul_rn(qz, qz)))));
}
// out of line for the rare exact paths
__device__ __noinline__ double4_32a plane_call(const double *off, unsigned ref, const double4_32a *__restrict__ sorted,
                                               const BoxDev *gp)
{
    double4_32a v;
    plane64(off, ref, sorted, gp, v.x, v.y, v.z, v.w);
    return v;
}
__device__ __noinline__ double4_32a vertex_exact(const CellSmem &S, unsigned tri,
                                                 const double4_32a *__restrict__ sorted, const BoxDev *gp)
{
    const double4_32a a = plane_call(S.off, S.pid[tri & 31u], sorted, gp);
    const double4_32a b = plane_call(S.off, S.pid[(tri >> 5) & 31u], sorted, gp);
    const double4_32a c = plane_call(S.off, S.pid[(tri >> 10) & 31u], sorted, gp);
    double4_32a v;
    solve64(a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y, c.z, c.w, v.x, v.y, v.z);
    v.w = 0.0;
    return v;
}

// A new vertex and its error bound, k_clip's bits (the gather threshold is
// formed from them, and the same candidates have to meet in a batch).
__device__ __forceinline__ float4 cell_vertex(const CellSmem &S, unsigned tri, const double4_32a *__restrict__ sorted,
                                              const BoxDev *gp)
{
    const float4 Pa = S.pf[tri & 31u], Pb = S.pf[(tri >> 5) & 31u], Pc = S.pf[tri >> 10];
    float x, y, z, er;
    solve32(Pa, Pb, Pc, plane_length(Pa.w), plane_length(Pb.w), plane_length(Pc.w), x, y, z, er);
    if (!(er < 1e30f)) {
        const double4_32a X = vertex_exact(S, tri, sorted, gp);
        rounded_vertex(X.x, X.y, X.z, x, y, z, er);
    }
    return make_float4(x, y, z, er);
}

// The margin rule of k_clip's plane test on the exact vertex and plane.
__device__ __noinline__ bool beyond_ref(const CellSmem &S, unsigned tri, unsigned ref,
                                        const double4_32a *__restrict__ sorted, const BoxDev *gp)
{
    const double4_32a v = vertex_exact(S, tri, sorted, gp), q = plane_call(S.off, ref, sorted, gp);
    return beyond64(q.x, q.y, q.z, __longlong_as_double(__double_as_longlong(q.w) + (1LL << 13)), v.x, v.y, v.z);
}

// Sort key of a candidate: |q|^2 / 2 in FP32 on a window of 16 binades above
// `base`, 26 bits, above the 6 bits of its place in the buffer.  Monotone in
// the exact |q|^2; equal upper bits are settled exactly (cand_before).
__device__ __forceinline__ unsigned cand_key(float half_d2, unsigned base)
{
    const unsigned b = __float_as_uint(half_d2);
    return min(b > base ? b - base : 0u, 0x7ffffffu) >> 1;
}

// Put the entries of a cell's sorted buffer whose key bits are equal in exact
// order (|q|^2, id, image code): each lane ranks its entries among those of
// the same key.  A tied candidate holds |q|^2 / 2 and its id in its plane's
// place meanwhile.  On exact lattices most entries are tied (runs of 8, 6, 12
// and 24 on a body-centred one); sorting a run by insertion on one lane, from
// the generators anew for each comparison, took most of the time there.
// Tessellation, insertion / rank (warp per cell): body-centred 2 x 16^3 0.51 /
// 0.33 ms (0.43), 2 x 40^3 4.65 / 2.42 (4.34), cubic 64^3 9.2 / 6.0 (15.1).
template <int G>
__device__ __noinline__ void settle_ties(CellSmem &S, int m, unsigned base, int gl,
                                         const double4_32a *__restrict__ sorted, const BoxDev *gp)
{
    unsigned char *const order = reinterpret_cast<unsigned char *>(S.tri);
    static_assert(sizeof(S.tri) >= CCB, "the new order fits in the new triangles' place");
    const auto key = [&](int e) { return cand_key(S.cf[S.perm[e]].w, base); };
    unsigned tied = 0;  // bit i: this lane's entry gl + G i
#pragma unroll 1
    for (int e = gl, i = 0; e < m; e += G, ++i) {
        const int v = S.perm[e];
        const unsigned kv = key(e);
        order[e] = (unsigned char)v;
        if (!((e > 0 && key(e - 1) == kv) || (e + 1 < m && key(e + 1) == kv))) continue;
        tied |= 1u << i;
        const unsigned ref = S.cid[v];
        const double o = plane_call(S.off, ref, sorted, gp).w;
        const int id = (int)__double_as_longlong(sorted[ref & IDX_MASK].w);
        S.cf[v].x = __int_as_float(__double2loint(o));
        S.cf[v].y = __int_as_float(__double2hiint(o));
        S.cf[v].z = __int_as_float(id);
    }
    __syncwarp();
    const auto before = [&](int u, int v) {  // buffer entries
        const float4 U = S.cf[u], V = S.cf[v];
        const unsigned long long du = (unsigned long long)__float_as_uint(U.y) << 32 | __float_as_uint(U.x),
                                 dv = (unsigned long long)__float_as_uint(V.y) << 32 | __float_as_uint(V.x);
        if (du != dv) return du < dv;
        if (__float_as_int(U.z) != __float_as_int(V.z)) return __float_as_int(U.z) < __float_as_int(V.z);
        return (S.cid[u] >> 27) < (S.cid[v] >> 27);
    };
#pragma unroll 1
    for (unsigned r = tied; r; r &= r - 1u) {
        const int e = gl + G * (__ffs((int)r) - 1), v = S.perm[e];
        const unsigned kv = key(e);
        int at = e;
#pragma unroll 1
        for (int j = e - 1; j >= 0 && key(j) == kv; --j) at -= before(v, S.perm[j]) ? 1 : 0;
#pragma unroll 1
        for (int j = e + 1; j < m && key(j) == kv; ++j) at += before(S.perm[j], v) ? 1 : 0;
        order[at] = (unsigned char)v;
    }
    __syncwarp();
#pragma unroll 1
    for (int e = gl, i = 0; e < m; e += G, ++i) {
        const int v = order[e];
        if ((tied >> i) & 1u) {  // (its entry is tied too: a run keeps its place)
            const double4_32a q = plane_call(S.off, S.cid[v], sorted, gp);
            S.cf[v].x = (float)q.x;
            S.cf[v].y = (float)q.y;
            S.cf[v].z = (float)q.z;
        }
        S.perm[e] = (unsigned char)v;
    }
    __syncwarp();
}

// Fill the holes a cut left beyond its new vertices from the end of the list
// (one lane per cell; a cut that swallows whole faces).
__device__ __noinline__ void fill_holes(CellSmem &S, int nnew, int nrem, int nt)
{
    unsigned long long holes = 0;
#pragma unroll 1
    for (int i = nnew; i < nrem; ++i) holes |= 1ull << S.hole[i];
#pragma unroll 1
    while (holes) {
        const int e = --nt;
        if (!((holes >> e) & 1ull)) {
            const int h = __ffsll((long long)holes) - 1;
            S.tf[h] = S.tf[e];
            S.vtri[h] = S.vtri[e];
            holes &= holes - 1ull;
        } else {
            holes &= ~(1ull << e);
        }
    }
}

// Generators per axis image of a bin index outside the grid (rare).
__device__ __noinline__ int2 wrap_bin(int b, int g)
{
    const int s = (b >= -g && b < 2 * g) ? (b < 0 ? -1 : (b >= g ? 1 : 0)) : floordiv(b, g);
    return make_int2(b - s * g, s);
}

__device__ __forceinline__ void order2(unsigned &a, unsigned &b)
{
    const unsigned lo = min(a, b), hi = max(a, b);
    a = lo;
    b = hi;
}

// Sort G * R keys held R per lane (key e = lane * R + r ascending) across the
// G lanes of a cell.
template <int G, int R>
__device__ __forceinline__ void sort_keys(unsigned (&key)[R], int gl)
{
    // each lane's own keys (odd-even merges)
#pragma unroll
    for (int p = 1; p < R; p <<= 1)
#pragma unroll
        for (int k = p; k >= 1; k >>= 1)
#pragma unroll
            for (int j = k % p; j + k < R; j += 2 * k)
#pragma unroll
                for (int i = 0; i < k; ++i)
                    if (i + j + k < R && (i + j) / (2 * p) == (i + j + k) / (2 * p)) order2(key[i + j], key[i + j + k]);
    // bitonic merges of runs of s lanes into runs of 2 s lanes
#pragma unroll 1
    for (int s = 1; s < G; s <<= 1) {
        const bool lower = (gl & s) == 0;
        unsigned o[R];
#pragma unroll
        for (int r = 0; r < R; ++r) o[r] = __shfl_xor_sync(FULL, key[R - 1 - r], 2 * s - 1);
#pragma unroll
        for (int r = 0; r < R; ++r) key[r] = lower ? min(key[r], o[r]) : max(key[r], o[r]);
#pragma unroll 1
        for (int j = s >> 1; j >= 1; j >>= 1) {
            const bool low = (gl & j) == 0;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const unsigned q = __shfl_xor_sync(FULL, key[r], j);
                key[r] = low ? min(key[r], q) : max(key[r], q);
            }
        }
#pragma unroll
        for (int j = R >> 1; j >= 1; j >>= 1)
#pragma unroll
            for (int r = 0; r < R; ++r)
                if ((r & j) == 0) order2(key[r], key[r | j]);
    }
}

// Keys of the buffered candidates, sorted, as a permutation; true if entries
// with equal key bits are left to settle.
template <int G, int R>
__device__ __forceinline__ bool sort_batch(CellSmem &S, int m, unsigned base, int gl)
{
    unsigned key[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int k = r * G + gl;
        key[r] = k < m ? (cand_key(S.cf[k].w, base) << 6) | (unsigned)k : 0xffffffffu;
    }
    sort_keys<G, R>(key, gl);
    bool tie = false;
    const unsigned nk = __shfl_down_sync(FULL, key[0], 1, G);
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int e = gl * R + r;
        S.perm[e] = (unsigned char)(key[r] & 63u);
        const unsigned next = r + 1 < R ? key[r + 1] : nk;
        tie |= e + 1 < m && (key[r] >> 6) == (next >> 6);
    }
    return tie;
}

// ---------------------------------------------------------------------------
// Geometry of a warp's cells once they are clipped.  Their planes, vertices
// and faces are spread over the 32 lanes as flat lists, because an FP64
// instruction occupies the pipe for the same 16 cycles whatever the number of
// active lanes: the FP64 work per cell is that of full warps.  Faces are taken
// in the order of their number of vertices, so that the lanes of a warp walk
// polygons of like length.
// ---------------------------------------------------------------------------
constexpr int GC = 32 / LANES;   // cells of a warp
constexpr int GV = 176;          // vertices of one pass (4 cells of 27; a fuller warp takes two passes)
constexpr int GP = 96;           // planes of one pass (4 cells of 16)
constexpr int TEAM = LANES;      // lanes of one cell
static_assert(GV >= CTM && GP >= CPM, "any one cell fits a pass");

struct __align__(16) GeomSmem {
    double vx[GV], vy[GV], vz[GV];
    double px[GP], py[GP], pz[GP], po[GP];  // planes, then face area and centroid
    double vp[GP];                          // pyramid volumes
    double off[GC][9];
    unsigned ref[GC][CPM];
    unsigned live[GC];                      // slots with a face
    int vbase[GC], pbase[GC];               // first vertex and plane of a cell in the lists
    int hist[16];
    unsigned short tri[GC][CTM];
    unsigned short item[GP], order[GP];     // cell << 5 | slot of a plane; planes by number of vertices
    unsigned short vitem[GV];               // cell << 6 | vertex
    unsigned char nxt[GP][CPM];             // vertex of the cell holding the directed edge plane -> slot
    unsigned char deg[GP];
    unsigned char bad[GC];
};
static_assert(sizeof(GeomSmem) <= GC * sizeof(CellSmem), "it takes the place of the clipped cells");
static_assert(offsetof(GeomSmem, nxt) % 16 == 0 && CPM % 16 == 0, "edge rows are read 16 bytes at a time");

__device__ __forceinline__ int plane_of(const GeomSmem &S, int c, unsigned slot)
{
    return S.pbase[c] + __popc(S.live[c] & ((1u << slot) - 1u));
}

// S holds the cells' references, triangles, offsets and live slots; w0 is the
// warp's first cell, nt this lane's cell's vertices (0: none to form).
__device__ __forceinline__ void
warp_geometry(GeomSmem &S, int lane, int64_t w0, int w, int nt, const BoxDev *gp, int self,
              const double4_32a *__restrict__ sorted, int64_t n, const BoxDev *__restrict__ boxes,
              const int *__restrict__ cbox, double *__restrict__ vol, double *__restrict__ cen, const Slots &sl,
              int *__restrict__ list, int *__restrict__ list_n)
{
    const int tc = lane / TEAM, tl = lane % TEAM;
    const int64_t sbase = (int64_t)self * MAXF, ns = n * (int64_t)MAXF;
    bool todo = nt > 0;
    while (__any_sync(FULL, todo)) {
        // ---- the cells of this pass: as many, in order, as the lists hold
        const int nl = __popc(S.live[tc]);
        int vb = todo && tl == 0 ? nt : 0, pb = todo && tl == 0 ? nl : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(FULL, vb, o), p = __shfl_up_sync(FULL, pb, o);
            if (lane >= o) { vb += v; pb += p; }
        }
        const bool mine = todo && vb <= GV && pb <= GP;  // prefix sums: true for a first run of the cells left
        const int nv = __reduce_max_sync(FULL, mine ? vb : 0), npl = __reduce_max_sync(FULL, mine ? pb : 0);
        vb -= nt;
        pb -= nl;
        if (mine && tl == 0) { S.vbase[tc] = vb; S.pbase[tc] = pb; }
        if (mine) {
            const unsigned lv = S.live[tc];
#pragma unroll 1
            for (unsigned r = lv; r; r &= r - 1u) {
                const int p = __ffs((int)r) - 1, k = pb + __popc(lv & ((1u << p) - 1u));
                if ((k & (TEAM - 1)) == tl) S.item[k] = (unsigned short)(tc << 5 | p);
            }
#pragma unroll 1
            for (int t = tl; t < nt; t += TEAM) S.vitem[vb + t] = (unsigned short)(tc << 6 | t);
        }
        if (lane < 16) S.hist[lane] = 0;
        {
            uint4 *const z = reinterpret_cast<uint4 *>(&S.nxt[0][0]);
#pragma unroll 1
            for (int i = lane; i < npl * CPM / 16; i += 32) z[i] = make_uint4(FULL, FULL, FULL, FULL);
        }
        __syncwarp();
        // ---- planes and edges
#pragma unroll 1
        for (int k = lane; k < npl; k += 32) {
            const int it = S.item[k], c = it >> 5;
            double x, y, z, o;
            plane64(S.off[c], S.ref[c][it & 31], sorted, boxes + cbox[w0 + c], x, y, z, o);
            S.px[k] = x; S.py[k] = y; S.pz[k] = z; S.po[k] = o;
            S.vp[k] = 0.0;
        }
#pragma unroll 1
        for (int k = lane; k < nv; k += 32) {
            const int it = S.vitem[k], c = it >> 6, t = it & 63;
            const unsigned v = S.tri[c][t], x = v & 31u, y = (v >> 5) & 31u, z = v >> 10;
            S.nxt[plane_of(S, c, x)][y] = (unsigned char)t;
            S.nxt[plane_of(S, c, y)][z] = (unsigned char)t;
            S.nxt[plane_of(S, c, z)][x] = (unsigned char)t;
        }
        __syncwarp();
        // ---- vertices; an edge two triangles claim is not a closed cell
#pragma unroll 1
        for (int k = lane; k < nv; k += 32) {
            const int it = S.vitem[k], c = it >> 6, t = it & 63;
            const unsigned v = S.tri[c][t], x = v & 31u, y = (v >> 5) & 31u, z = v >> 10;
            const int a = plane_of(S, c, x), b = plane_of(S, c, y), d = plane_of(S, c, z);
            if (S.nxt[a][y] != t || S.nxt[b][z] != t || S.nxt[d][x] != t) S.bad[c] = 1;
            vertex64(S, a, b, d, S.vx[k], S.vy[k], S.vz[k]);
        }
        // ---- faces by number of vertices: the bytes of the edge row in use
#pragma unroll 1
        for (int k = lane; k < npl; k += 32) {
            const uint4 *const r = reinterpret_cast<const uint4 *>(S.nxt[k]);
            const uint4 a = r[0], b = r[1];
            const unsigned u = ~a.x & 0x80808080u, v = ~a.y & 0x80808080u, x = ~a.z & 0x80808080u, y = ~a.w & 0x80808080u;
            const unsigned u2 = ~b.x & 0x80808080u, v2 = ~b.y & 0x80808080u, x2 = ~b.z & 0x80808080u, y2 = ~b.w & 0x80808080u;
            const int d = min(__popc(u | v >> 1 | x >> 2 | y >> 3 | u2 >> 4 | v2 >> 5 | x2 >> 6 | y2 >> 7), 15);
            S.deg[k] = (unsigned char)d;
            atomicAdd(&S.hist[d], 1);
        }
        __syncwarp();
        {
            const int h = lane < 16 ? S.hist[15 - lane] : 0;  // most vertices first
            int p = h;
#pragma unroll
            for (int o = 1; o < 16; o <<= 1) {
                const int q = __shfl_up_sync(FULL, p, o);
                if (lane >= o) p += q;
            }
            if (lane < 16) S.hist[15 - lane] = p - h;
        }
        __syncwarp();
#pragma unroll 1
        for (int k = lane; k < npl; k += 32) S.order[atomicAdd(&S.hist[S.deg[k]], 1)] = (unsigned short)k;
        __syncwarp();
#pragma unroll 1
        for (int j = lane; j < npl; j += 32) {
            const int k = S.order[j], it = S.item[k], c = it >> 5;
            const unsigned p = it & 31;
            const int vbc = S.vbase[c];
            // the walk starts at the vertex holding the edge to the lowest slot
            unsigned y = 0;
            int t0 = 255;
            {
                const uint4 *const r = reinterpret_cast<const uint4 *>(S.nxt[k]);
                const uint4 a = r[0], b = r[1];
                const unsigned wv[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
                for (int q = 7; q >= 0; --q) {
                    const unsigned u = ~wv[q] & 0x80808080u;
                    if (u) {
                        const int s = __ffs((int)u) >> 3;  // byte 0..3 (its bit 7 is set)
                        y = (unsigned)(4 * q + s - 1);
                        t0 = (int)((wv[q] >> (8 * (s - 1))) & 255u);
                    }
                }
            }
            const double qx = S.px[k], qy = S.py[k], qz = S.pz[k];
            const int ka = fan_axis(qx, qy, qz);
            const double *T1 = (ka == 0 ? S.vy : S.vx) + vbc, *T2 = (ka == 2 ? S.vy : S.vz) + vbc;
            const double u0 = T1[t0], v0 = T2[t0];
            FaceFan F;
            bool ok = false, any = false;
#pragma unroll 1
            for (int guard = 0; guard < CTM; ++guard) {
                const unsigned vt = S.tri[c][guard == 0 ? t0 : (int)S.nxt[k][y]];
                y = (vt & 31u) ^ ((vt >> 5) & 31u) ^ (vt >> 10) ^ p ^ y;
                const int tn = S.nxt[k][y];
                if (tn == 255) break;
                if (tn == t0) { ok = true; break; }
                const double bu = T1[tn] - u0, bv = T2[tn] - v0;
                if (any) F.edge(bu, bv);
                else F.begin(bu, bv);
                any = true;
            }
            if (!ok) S.bad[c] = 1;
            double area, fx, fy, fz, vp;
            face_of_fan(F, ka, qx, qy, qz, S.po[k], S.vx[vbc + t0], S.vy[vbc + t0], S.vz[vbc + t0], area, fx, fy, fz, vp);
            S.px[k] = area; S.py[k] = fx; S.pz[k] = fy; S.po[k] = fz;
            S.vp[k] = vp;
        }
        __syncwarp();
        // ---- slots, cell by cell in order of the planes
        const double amin = gp->amin;
        int nface = 0;
        {
            const int nout = mine && !S.bad[tc] ? nl : 0, maxout = __reduce_max_sync(FULL, nout);
#pragma unroll 1
            for (int i = tl; i - tl < maxout; i += TEAM) {
                const int k = pb + i;
                double area = 0.0, fx = 0.0, fy = 0.0, fz = 0.0;
                if (i < nout) {
                    // the first moment takes the centroid's place
                    const double vw = __dmul_rn(0.75, S.vp[k]);
                    area = S.px[k]; fx = S.py[k]; fy = S.pz[k]; fz = S.po[k];
                    S.py[k] = __dmul_rn(vw, fx);
                    S.pz[k] = __dmul_rn(vw, fy);
                    S.po[k] = __dmul_rn(vw, fz);
                }
                const bool keep = i < nout && abs_bits(area) > abs_bits(amin);
                const unsigned km = (__ballot_sync(FULL, keep) >> (tc * TEAM)) & ((1u << TEAM) - 1u);
                if (keep) {
                    const int64_t s = sbase + nface + __popc(km & ((1u << tl) - 1u));
                    const unsigned ref = S.ref[tc][S.item[k] & 31], code = ref >> 27;
                    int nb = self, sh;
                    if (code == 31u) {
                        const int kf = (int)(ref & 7u), d = kf >> 1, e = d == 0 ? 1 : (d == 1 ? 3 : 9);
                        sh = 13 + ((kf & 1) ? -e : e);
                    } else {
                        nb = (int)__double_as_longlong(sorted[ref & IDX_MASK].w);
                        sh = (int)code;
                    }
                    sl.nb[s] = nb;
                    sl.sh[s] = (unsigned char)sh;
                    sl.area[s] = area;
                    sl.fc[s] = fx;
                    sl.fc[ns + s] = fy;
                    sl.fc[2 * ns + s] = fz;
                }
                nface += __popc(km);
            }
        }
        __syncwarp();
        // ---- volume and first moment: k_clip's tree over the 32 slots (p and
        // p + 16, then p + 8, p + 4, p + 2, p + 1; a slot without a face adds 0)
        double a0, a1, a2, a3;
        {
            const unsigned lv = S.live[tc];
            a0 = a1 = a2 = a3 = 0.0;
#pragma unroll 1
            for (int p = tl; p < 16; p += 8) {
                const bool lo = mine && ((lv >> p) & 1u), hi = mine && ((lv >> (p + 16)) & 1u);
                const int k = lo ? pb + __popc(lv & ((1u << p) - 1u)) : 0;
                const int h = hi ? pb + __popc(lv & ((1u << (p + 16)) - 1u)) : 0;
                const double b0 = __dadd_rn(lo ? S.vp[k] : 0.0, hi ? S.vp[h] : 0.0);
                const double b1 = __dadd_rn(lo ? S.py[k] : 0.0, hi ? S.py[h] : 0.0);
                const double b2 = __dadd_rn(lo ? S.pz[k] : 0.0, hi ? S.pz[h] : 0.0);
                const double b3 = __dadd_rn(lo ? S.po[k] : 0.0, hi ? S.po[h] : 0.0);
                a0 = __dadd_rn(a0, b0);  // (0 + b is b)
                a1 = __dadd_rn(a1, b1);
                a2 = __dadd_rn(a2, b2);
                a3 = __dadd_rn(a3, b3);
            }
        }
        // each exchange halves the sums a lane keeps: lanes 0-1 of the eight end
        // with the volume, 2-3, 4-5 and 6-7 with the moment's components
        static_assert(TEAM == 8, "three exchanges");
        {
            const bool h4 = (tl & 4) != 0, h2 = (tl & 2) != 0;
            double k0 = h4 ? a2 : a0, k1 = h4 ? a3 : a1;
            const double s0 = h4 ? a0 : a2, s1 = h4 ? a1 : a3;
            k0 += __shfl_xor_sync(FULL, s0, 4);
            k1 += __shfl_xor_sync(FULL, s1, 4);
            double q = h2 ? k1 : k0;
            q += __shfl_xor_sync(FULL, h2 ? k0 : k1, 2);
            q += __shfl_xor_sync(FULL, q, 1);
            a0 = q;
        }
        if (mine && (tl & 1) == 0) {
            if (S.bad[tc]) {
                if (tl == 0) list[atomicAdd(list_n, 1)] = w;
            } else if (tl == 0) {
                sl.cnt[self] = nface;
                vol[self] = a0;
            } else {
                cen[(tl / 2 - 1) * n + self] = a0;
            }
        }
        todo = todo && !mine;
        __syncwarp();
    }
}

// Largest |v|^2 bound of a cell's vertices (vertex_r2).
// Formed when candidates are gathered or screened, not at every cut.
template <int G>
__device__ __forceinline__ float r2_max(const CellSmem &S, int nt, int gl)
{
    float mr = 0.0f;
#pragma unroll 1
    for (int t = gl; t < nt; t += G) {
        const float4 V = S.tf[t];
        // (a corner of the starting box has no error; the factors are k_clip's, so
        // that the same candidates are gathered)
        mr = fmaxf(mr, vertex_r2(V.x, V.y, V.z, V.w) * (V.w == 0.0f ? 1.000001f : 1.00001f));
    }
#pragma unroll
    for (int o = G / 2; o >= 1; o >>= 1) mr = fmaxf(mr, __shfl_xor_sync(FULL, mr, o));
    return mr;
}

template <int G>
__global__ void __launch_bounds__(64, 8)
k_cells(const double4_32a *__restrict__ sorted, const float4 *__restrict__ sortedf, const int *__restrict__ start,
        int64_t n, const BoxDev *__restrict__ boxes, const int *__restrict__ cbox, double *__restrict__ vol,
        double *__restrict__ cen, Slots sl, int cand_cap, int *__restrict__ list, int *__restrict__ list_n)
{
    constexpr int CPW = 32 / G;
    constexpr unsigned GM = (1u << G) - 1u;
    extern __shared__ __align__(16) unsigned char dyn_smem[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int gl = lane & (G - 1), gsh = lane & ~(G - 1);
    const unsigned ltg = (1u << gl) - 1u;
    const int64_t w0 = ((int64_t)blockIdx.x * (blockDim.x >> 5) + wid) * CPW;
    if (w0 >= n) return;
    const int64_t wi = w0 + gsh / G;
    const int w = (int)(wi < n ? wi : n - 1);  // a group past n repeats the last cell and writes nothing
    CellSmem &S = reinterpret_cast<CellSmem *>(dyn_smem)[wid * CPW + gsh / G];
    const BoxDev *const gp = boxes + cbox[w];
    const auto gball = [&](bool p) { return (__ballot_sync(FULL, p) >> gsh) & GM; };

    // ---- starting box (as in k_clip)
    if (gl < 6) {
        const int d = gl >> 1;
        const float Lf = gp->Lf[d], sLf = (gl & 1) ? -Lf : Lf;
        const double L = gp->L[d];
        const float fo = (float)half_of(__double_as_longlong(__dmul_rn(L, L)));
        S.pf[gl] = make_float4(d == 0 ? sLf : 0.0f, d == 1 ? sLf : 0.0f, d == 2 ? sLf : 0.0f, fo);
        S.pid[gl] = BOX_PLANE | (unsigned)gl;
    }
#pragma unroll 1
    for (int k = gl; k < 9; k += G) {
        const int d = k / 3, s = k - 3 * d;
        const double p = d == 0 ? sorted[w].x : (d == 1 ? sorted[w].y : sorted[w].z);
        const double L = gp->L[d];
        const double o = s == 1 ? -p : (s == 0 ? -L - p : L - p);
        S.off[k] = o;
        S.offf[k] = (float)o;
    }
    float lim4;  // at least 4 r_max^2
    float slack, bs0, bs1, bs2, lo0, lo1, lo2, hi0, hi1, hi2;  // distances from p to its bin's walls, less the slack
    int cb0, cb1, cb2;
    const int g0 = gp->g[0], g1 = gp->g[1], g2 = gp->g[2], bin_off = gp->bin_off;
    {
        const float L0 = gp->Lf[0], L1 = gp->Lf[1], L2 = gp->Lf[2];
        if (gl < 8) {
            const int sx = gl & 1, sy = (gl >> 1) & 1, sz = (gl >> 2) & 1;
            unsigned a = sx, b = 2 + sy, c = 4 + sz;
            if ((sx ^ sy ^ sz) & 1) { const unsigned t = b; b = c; c = t; }
            const float x = 0.5f * (sx ? -L0 : L0), y = 0.5f * (sy ? -L1 : L1), z = 0.5f * (sz ? -L2 : L2);
            S.tf[gl] = make_float4(x, y, z, 0.0f);
            S.vtri[gl] = (unsigned short)(a | (b << 5) | (c << 10));
        }
        lim4 = fmaf(L0, L0, fmaf(L1, L1, L2 * L2)) * 1.000001f;
        slack = 2e-6f * fmaxf(L0, fmaxf(L1, L2));
        bs0 = gp->bsf[0]; bs1 = gp->bsf[1]; bs2 = gp->bsf[2];
        const float4 mf = sortedf[w];
        const auto home = [&](float p, float ib, float bs, int g, int &cb, float &lo, float &hi) {
            const int c = (int)floorf(p * ib);
            cb = c < 0 ? 0 : (c >= g ? g - 1 : c);
            lo = p - (float)cb * bs - slack;
            hi = (float)(cb + 1) * bs - p - slack;
        };
        home(mf.x, gp->ibsf[0], bs0, g0, cb0, lo0, hi0);
        home(mf.y, gp->ibsf[1], bs1, g1, cb1, lo1, hi1);
        home(mf.z, gp->ibsf[2], bs2, g2, cb2, lo2, hi2);
    }
#pragma unroll 1
    for (int r = gl; r < CPM; r += G) S.bm[r] = 0u;
    // key window: from 2^-10 of a squared bin edge upwards
    const unsigned kbase = max(__float_as_uint(bs0 * bs0), 10u << 23) - (10u << 23);
    __syncwarp();

    int np = 6, nt = 8;
    float limk = __int_as_float(0x7f800000), limlow = lim4;  // gather threshold, smallest lim4 so far
    bool bad = false, done = wi >= n;
    int ncand = 0, rh = 1, chunk = 0, chunk_end = SHELLS.first[2];
    int nbin = 0, depth = 0, step = 0;  // bins of the chunk with generators left, their largest count, the next entry

    while (!__all_sync(FULL, done)) {
        // ---- gather (the batches of k_clip: one entry of each of 32 bins a step)
        bool ring_done = false, want = !done;
        for (;;) {
            const bool any = step < depth;
            bool act = want && ncand + 32 <= cand_cap;
            if (act && !any && chunk >= chunk_end) { ring_done = true; want = false; act = false; }
            if (!__any_sync(FULL, act)) break;
            const bool setup = act && !any;
            if (__any_sync(FULL, setup)) {
                // the chunk's bins that hold generators within reach, in order
                const float reach = 1.02f * fmaf(slack, sqrt_fast(limk), limk);
                const int b0 = SHELLS.chunk[chunk], nb = setup ? SHELLS.chunk[chunk + 1] - b0 : 0;
                const int maxnb = __reduce_max_sync(FULL, nb);
                int found = 0, most = 0;
#pragma unroll 1
                for (int i = gl; i - gl < maxnb; i += G) {
                    int cnt = 0, first = 0;
                    unsigned code = 0;
                    if (i < nb) {
                        const unsigned e = SHELLS.bin[b0 + i];
                        const int ox = (int)(e & 15u) - 8, oy = (int)((e >> 4) & 15u) - 8, oz = (int)(e >> 8) - 8;
                        // nearest point of the bin: a bin beyond the threshold has
                        // nothing to keep (1 %: the threshold may still grow by rounding)
                        const float dx = ox == 0 ? 0.0f : fmaxf(ox > 0 ? fmaf((float)(ox - 1), bs0, hi0) : fmaf((float)(-ox - 1), bs0, lo0), 0.0f);
                        const float dy = oy == 0 ? 0.0f : fmaxf(oy > 0 ? fmaf((float)(oy - 1), bs1, hi1) : fmaf((float)(-oy - 1), bs1, lo1), 0.0f);
                        const float dz = oz == 0 ? 0.0f : fmaxf(oz > 0 ? fmaf((float)(oz - 1), bs2, hi2) : fmaf((float)(-oz - 1), bs2, lo2), 0.0f);
                        if (fmaf(dx, dx, fmaf(dy, dy, dz * dz)) <= reach) {
                            int bx = cb0 + ox, by = cb1 + oy, bz = cb2 + oz, shx = 0, shy = 0, shz = 0;
                            if ((unsigned)bx >= (unsigned)g0) { const int2 v = wrap_bin(bx, g0); bx = v.x; shx = v.y; }
                            if ((unsigned)by >= (unsigned)g1) { const int2 v = wrap_bin(by, g1); by = v.x; shy = v.y; }
                            if ((unsigned)bz >= (unsigned)g2) { const int2 v = wrap_bin(bz, g2); bz = v.x; shz = v.y; }
                            // images two or more boxes away never cut
                            if (max(abs(shx), max(abs(shy), abs(shz))) <= 1) {
                                const int b = bin_off + bx + g0 * (by + g1 * bz);
                                first = start[b];
                                cnt = start[b + 1] - first;
                                code = (unsigned)(shx + 1) | (unsigned)(shy + 1) << 2 | (unsigned)(shz + 1) << 4 |
                                       (abs(shx) + abs(shy) + abs(shz) <= 1 ? 64u : 0u);
                            }
                        }
                    }
                    if (cnt > 31) { bad = true; cnt = 0; }  // a crowded bin: k_clip's cell
                    const unsigned km = gball(cnt > 0);
                    if (cnt > 0) {
                        const int k = found + __popc(km & ltg);
                        S.bin[k] = (unsigned)first | ((unsigned)cnt << 27);
                        S.bcode[k] = (unsigned char)code;
                    }
                    found += __popc(km);
                    most = max(most, cnt);
                }
#pragma unroll
                for (int o = G / 2; o >= 1; o >>= 1) most = max(most, __shfl_xor_sync(FULL, most, o));
                if (setup) {
                    nbin = found;
                    depth = most;
                    step = 0;
                    ++chunk;
                }
                __syncwarp();
                continue;
            }
            const int maxbin = __reduce_max_sync(FULL, act ? nbin : 0);
#pragma unroll 1
            for (int i = gl; i - gl < maxbin; i += G) {
                bool keep = false;
                unsigned ref = 0;
                if (act && i < nbin) {
                    const unsigned b = S.bin[i], code = S.bcode[i];
                    if (step < (int)(b >> 27)) {
                        const unsigned idx = (b & IDX_MASK) + (unsigned)step;
                        const float4 Pf = sortedf[idx];
                        const unsigned sx = code & 3u, sy = (code >> 2) & 3u, sz = (code >> 4) & 3u;
                        const float qx = Pf.x + S.offf[sx], qy = Pf.y + S.offf[3 + sy], qz = Pf.z + S.offf[6 + sz];
                        const float d2f = fmaf(qx, qx, fmaf(qy, qy, qz * qz));
                        keep = !(idx == (unsigned)w && (code >> 6)) && d2f <= limk;
                        ref = idx | ((sx + 3u * sy + 9u * sz) << 27);
                    }
                }
                const unsigned km = gball(keep);
                if (keep) S.cid[ncand + __popc(km & ltg)] = ref;
                ncand += __popc(km);
            }
            if (act) ++step;
        }
        __syncwarp();

        // ---- flush: planes, order, clip
        const int m = done ? 0 : ncand;
        const int maxm = __reduce_max_sync(FULL, m);
        bool coincident = bad;
#pragma unroll 1
        for (int k = gl; k < m; k += G) {
            double qx, qy, qz, o;
            plane64(S.off, S.cid[k], sorted, gp, qx, qy, qz, o);
            S.cf[k] = make_float4((float)qx, (float)qy, (float)qz, (float)o);
            coincident |= __double_as_longlong(o) == 0;
        }
        bad = gball(coincident) != 0u;
        __syncwarp();
        if (maxm > 0) {
            const bool tie = maxm <= 32 ? sort_batch<G, 32 / G>(S, m, kbase, gl) : sort_batch<G, 64 / G>(S, m, kbase, gl);
            const bool gtie = gball(tie) != 0u;
            __syncwarp();
            if (__any_sync(FULL, gtie)) settle_ties<G>(S, gtie ? m : 0, kbase, gl, sorted, gp);
        }
        // Candidates before `fit` are tried one by one; the rest are first
        // screened, a candidate to a lane, against the cell as it is by then: the
        // cell only shrinks, so one that cuts nothing now never will.  The
        // first SCREEN of a new cell mostly cut and are not screened.
        int k = 0, mc = m, fit = np == 6 ? min(m, SCREEN) : 0;
        bool run = !done && !bad;
        const float rmax = sqrt_fast(0.25f * lim4) * 1.01f;  // |v| of every vertex to come (limlow below)
#pragma unroll 1
        while (__any_sync(FULL, run && k < mc)) {
            const bool scr = run && k >= fit && k < mc;
            if (__any_sync(FULL, scr)) {
                {
                    const float r2 = r2_max<G>(S, nt, gl);
                    if (np > 6) lim4 = 4.0f * r2;
                }
                const int cnt = scr ? mc - k : 0, maxc = __reduce_max_sync(FULL, cnt);
                int dst = k;
#pragma unroll 1
                for (int i = 0; i < maxc; i += G) {
                    bool keep = false;
                    const int kc = i + gl < cnt ? (int)S.perm[k + i + gl] : 0;
                    if (i + gl < cnt) {
                        const float4 F = S.cf[kc];
                        if (2.0f * F.w <= lim4 * 1.000001f) {
                            const float qn = sqrt_fast(2.0f * F.w) * 1.00003f;
                            float far = -__int_as_float(0x7f800000);
#pragma unroll 1
                            for (int t = 0; t < nt; ++t) {
                                const float4 V = S.tf[t];
                                const float s = fmaf(F.x, V.x, fmaf(F.y, V.y, fmaf(F.z, V.z, -F.w)));
                                far = fmaxf(far, fmaf(qn, V.w, s));
                            }
                            // (one rounding more than the test below: 17 u for 16 u)
                            keep = !(far < -17.0f * 5.9604645e-8f * 1.0001f * fmaf(qn, rmax, F.w)) || !(F.w > 1e-30f);
                        }
                    }
                    const unsigned km = gball(keep);
                    __syncwarp();
                    if (keep) S.perm[dst + __popc(km & ltg)] = (unsigned char)kc;
                    dst += __popc(km);
                }
                if (scr) { mc = dst; fit = dst; }
                __syncwarp();
            }
            // find the next candidate that cuts
            unsigned my = 0;  // bit c: this lane's vertex c G + gl is beyond
            bool search = run && k < fit;
            int kk = 0;
#pragma unroll 1
            while (__any_sync(FULL, search)) {
                unsigned um = 0;
                if (search) {
                    kk = S.perm[k];
                    const float4 F = S.cf[kk];
                    if (2.0f * F.w > lim4 * 1.000001f) {
                        k = mc;  // this and every later candidate is out of reach
                    } else {
                        // |s - exact| <= |q| err + 16 u (|q||v| + o) for every vertex
                        const float qn = sqrt_fast(2.0f * F.w) * 1.00003f;
                        const float cst = F.w > 1e-30f ? 16.0f * 5.9604645e-8f * 1.0001f * fmaf(qn, rmax, F.w)
                                                       : __int_as_float(0x7f800000);
                        unsigned bit = 1u;
#pragma unroll 1
                        for (int t = gl; t < nt; t += G, bit <<= 1) {
                            const float4 V = S.tf[t];
                            const float s = fmaf(F.x, V.x, fmaf(F.y, V.y, fmaf(F.z, V.z, -F.w)));
                            const float B = fmaf(qn, V.w, cst);
                            if (s > B) my |= bit;
                            else if (!(s < -B)) um |= bit;
                        }
                    }
                }
                if (__any_sync(FULL, um != 0u)) {
#pragma unroll 1
                    while (um) {
                        const int c = __ffs((int)um) - 1;
                        um &= um - 1u;
                        if (beyond_ref(S, S.vtri[c * G + gl], S.cid[kk], sorted, gp)) my |= 1u << c;
                    }
                    __syncwarp();
                }
                const bool hit = gball(my != 0u) != 0u;
                if (search && !hit) ++k;
                search = search && !hit && k < fit;
            }
            bool go = gball(my != 0u) != 0u;
            if (!__any_sync(FULL, go)) continue;
            // the removed triangles and their directed edges
            int pos = __popc(my);
            {
                const int c = pos;
#pragma unroll
                for (int o = 1; o < G; o <<= 1) {
                    const int v = __shfl_up_sync(FULL, pos, o, G);
                    if (gl >= o) pos += v;
                }
                pos -= c;
            }
            const int nrem = __shfl_sync(FULL, pos + __popc(my), G - 1, G);
            bool over = go && nrem > CNS;
#pragma unroll 1
            while (my) {
                const int t = (__ffs((int)my) - 1) * G + gl;
                my &= my - 1u;
                const unsigned v = S.vtri[t];
                if (pos < CNS) S.hole[pos] = (unsigned char)t;
                ++pos;
                const unsigned x = v & 31u, y = (v >> 5) & 31u, z = v >> 10;
                atomicOr(&S.bm[x], 1u << y);
                atomicOr(&S.bm[y], 1u << z);
                atomicOr(&S.bm[z], 1u << x);
            }
            const bool cut = go;
            // plane slot: a fresh one while there is one, else one no vertex refers to
            int kp = np;
            if (__any_sync(FULL, go && np >= CPM)) {
                unsigned live = 0;
#pragma unroll 1
                for (int t = gl; t < nt; t += G) {
                    const unsigned v = S.vtri[t];
                    live |= (1u << (v & 31u)) | (1u << ((v >> 5) & 31u)) | (1u << (v >> 10));
                }
#pragma unroll
                for (int o = G / 2; o >= 1; o >>= 1) live |= __shfl_xor_sync(FULL, live, o);
                if (np >= CPM) {
                    kp = __ffs((int)~live) - 1;
                    if (kp < 0) { over |= go; kp = 0; }
                }
            }
            go = go && !over;
            if (go && gl == 0) {
                S.pf[kp] = S.cf[kk];
                S.pid[kp] = S.cid[kk];
            }
            __syncwarp();
            // rim edges: removed x -> y whose reverse is not removed
            int nnew = 0;
            unsigned xs = 0, ys = 0;
            const int maxrem = __reduce_max_sync(FULL, go ? nrem : 0);
#pragma unroll 1
            for (int i = gl; i - gl < maxrem; i += G) {
                unsigned x = 0, y = 0, z = 0;
                bool f0 = false, f1 = false, f2 = false;
                if (go && i < nrem) {
                    const unsigned v = S.vtri[S.hole[i]];
                    x = v & 31u, y = (v >> 5) & 31u, z = v >> 10;
                    f0 = !((S.bm[y] >> x) & 1u);
                    f1 = !((S.bm[z] >> y) & 1u);
                    f2 = !((S.bm[x] >> z) & 1u);
                    if (f0) { xs |= 1u << x; ys |= 1u << y; }
                    if (f1) { xs |= 1u << y; ys |= 1u << z; }
                    if (f2) { xs |= 1u << z; ys |= 1u << x; }
                }
                const int cnt = (int)f0 + (int)f1 + (int)f2;
                const unsigned b0 = gball(cnt & 1), b1 = gball(cnt & 2);
                int o = nnew + __popc(b0 & ltg) + 2 * __popc(b1 & ltg);
                const unsigned h = (unsigned)kp << 10;
                if (f0) { if (o < CNS) S.tri[o] = (unsigned short)(x | (y << 5) | h); ++o; }
                if (f1) { if (o < CNS) S.tri[o] = (unsigned short)(y | (z << 5) | h); ++o; }
                if (f2) { if (o < CNS) S.tri[o] = (unsigned short)(z | (x << 5) | h); ++o; }
                nnew += __popc(b0) + 2 * __popc(b1);
            }
            __syncwarp();
            if (cut)
#pragma unroll
                for (int r = 0; r < CPM / G; ++r) S.bm[r * G + gl] = 0u;
#pragma unroll
            for (int o = G / 2; o >= 1; o >>= 1) {
                xs |= __shfl_xor_sync(FULL, xs, o);
                ys |= __shfl_xor_sync(FULL, ys, o);
            }
            over |= go && (nnew > CNS || nnew < 3 || xs != ys || __popc(xs) != nnew || nt - nrem + nnew > CTM);
            if (over) { bad = true; run = false; go = false; }
            // the new vertices, in the removed ones' places and after the last
            const int maxnew = __reduce_max_sync(FULL, go ? nnew : 0);
#pragma unroll 1
            for (int i = gl; i - gl < maxnew; i += G) {
                if (go && i < nnew) {
                    const unsigned v = S.tri[i];
                    const int t = i < nrem ? (int)S.hole[i] : nt + i - nrem;
                    S.tf[t] = cell_vertex(S, v, sorted, gp);
                    S.vtri[t] = (unsigned short)v;
                }
            }
            __syncwarp();
            if (__any_sync(FULL, go && nnew < nrem)) {
                if (go && nnew < nrem && gl == 0) fill_holes(S, nnew, nrem, nt);
                __syncwarp();
            }
            if (go) {
                nt += nnew - nrem;
                np = max(np, kp + 1);
                ++k;
            }
        }
        {
            const float r2 = r2_max<G>(S, nt, gl);
            if (np > 6) lim4 = 4.0f * r2;
        }
        // bins are passed over, and rmax bounds |v|, by an earlier limit: it may
        // not grow past their margins (it shrinks but for the error bounds)
        limlow = fminf(limlow, lim4);
        if (lim4 > 1.005f * limlow) bad = true;
        if (np > 6) limk = fmaf(lim4, 1.00001f, slack * sqrtf(lim4));
        if (!done) {
            ncand = 0;
            if (bad) {
                done = true;
            } else if (ring_done) {
                const float rr = (float)rh;
                const float R = fmaxf(fminf(fminf(fmaf(rr, bs0, fminf(lo0, hi0)), fmaf(rr, bs1, fminf(lo1, hi1))),
                                            fmaf(rr, bs2, fminf(lo2, hi2))), 0.0f);
                if (lim4 <= R * R * 0.999999f) {
                    done = true;
                } else if (++rh > CELL_RINGS) {
                    bad = true;
                    done = true;
                } else {
                    chunk_end = SHELLS.first[rh + 1];
                }
            }
        }
        __syncwarp();
    }

    // ---- the cells' topology, in the same memory, and their geometry
    const int self = (int)__double_as_longlong(sorted[w].w);
    if (wi >= n) nt = 0;
    if (bad && nt > 0) {
        if (gl == 0) list[atomicAdd(list_n, 1)] = w;
        nt = 0;
    }
    GeomSmem &T = *reinterpret_cast<GeomSmem *>(dyn_smem + (size_t)wid * CPW * sizeof(CellSmem));
    {
        constexpr int NP = CPM / G, NV = CTM / G;
        unsigned ref[NP], tri[NV], lv = 0;
        const double off0 = S.off[gl], off8 = S.off[8];
#pragma unroll
        for (int r = 0; r < NP; ++r) ref[r] = S.pid[r * G + gl];
#pragma unroll
        for (int r = 0; r < NV; ++r) {
            const unsigned v = S.vtri[r * G + gl];
            tri[r] = v;
            if (r * G + gl < nt) lv |= (1u << (v & 31u)) | (1u << ((v >> 5) & 31u)) | (1u << (v >> 10));
        }
#pragma unroll
        for (int o = G / 2; o >= 1; o >>= 1) lv |= __shfl_xor_sync(FULL, lv, o);
        __syncwarp();
        const int c = gsh / G;
        T.off[c][gl] = off0;
#pragma unroll
        for (int r = 0; r < NP; ++r) T.ref[c][r * G + gl] = ref[r];
#pragma unroll
        for (int r = 0; r < NV; ++r) T.tri[c][r * G + gl] = (unsigned short)tri[r];
        if (gl == 0) {
            T.off[c][8] = off8;
            T.live[c] = lv;
            T.bad[c] = 0;
        }
        __syncwarp();
    }
    warp_geometry(T, lane, w0, w, nt, gp, self, sorted, n, boxes, cbox, vol, cen, sl, list, list_n);
}

}  // namespace

void launch_cells(const double4_32a *sorted, const float4 *sortedf, const int *start, int64_t n, const BoxDev *boxes,
                  const int *cbox, int cand_cap, double *vol, double *cen, Slots sl, int *list, int *list_n,
                  cudaStream_t s)
{
    constexpr int WARPS = 2, CELLS = WARPS * 32 / LANES;
    constexpr size_t smem = sizeof(CellSmem) * CELLS;
    static_assert(smem <= 48 * 1024, "no opt-in needed");
    cand_cap = cand_cap < 32 ? 32 : (cand_cap > CCB ? CCB : cand_cap);
    k_cells<LANES><<<(unsigned)((n + CELLS - 1) / CELLS), 32 * WARPS, smem, s>>>(sorted, sortedf, start, n, boxes, cbox,
                                                                                vol, cen, sl, cand_cap, list, list_n);
}

}  // namespace mm
