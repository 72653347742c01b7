"""The two clippers form the same FP32 vertex and error bound, bit for bit: the
security limit and with it the candidates that meet in a batch hang on them,
and a box stepped alone (warp-per-cell clipper below 4096 cells) has to give
the cells it gives in a larger batch (grouped clipper)."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_1707_05333_gb300 import build as BD

pytestmark = pytest.mark.gpu

PROBE = r"""
#include "mm_cells.cu"
#include "mm_clip.cu"
using namespace mm;
// 32 planes a block (the bisectors between the block's generator and the 32
// after it), each thread 64 triples of them; out: vertex, bound, |v|^2 bound
__global__ void k_probe(const double4_32a *gen, float *cells, float *clip)
{
    __shared__ CellSmem A;
    __shared__ ClipSmem<1, CapMain> B;
    const double4_32a *const g = gen + 33 * blockIdx.x;
    const int t = threadIdx.x;
    if (t < 9) {
        const int d = t / 3;
        A.off[t] = -(d == 0 ? g[0].x : (d == 1 ? g[0].y : g[0].z));
    }
    __syncthreads();
    {
        const unsigned ref = (unsigned)(33 * blockIdx.x + 1 + t) | (13u << 27);
        double x, y, z, o;
        plane64(A.off, ref, gen, nullptr, x, y, z, o);
        A.pid[t] = ref;
        A.pf[t] = B.pf[t] = make_float4((float)x, (float)y, (float)z, (float)o);
        B.pfn[t] = plane_length((float)o);
        B.px[t] = x; B.py[t] = y; B.pz[t] = z; B.po[t] = o;
    }
    __syncthreads();
    for (int k = 0; k < 64; ++k) {
        const int a = t, b = (t + 1 + k % 31) & 31, c = (b + 1 + (5 * k + t) % 29) & 31;
        if (a == b || b == c || a == c) continue;
        const float4 u = cell_vertex(A, (unsigned)(a | b << 5 | c << 10), gen, nullptr);
        float4 v;
        long long r2;
        double X, Y, Z;
        new_vertex<1>(B, (unsigned)(a | b << 8), c, r2, X, Y, Z, v);
        const long i = 5 * (64 * (32 * (long)blockIdx.x + t) + k);
        cells[i] = u.x; cells[i + 1] = u.y; cells[i + 2] = u.z; cells[i + 3] = u.w;
        cells[i + 4] = vertex_r2(u.x, u.y, u.z, u.w) * 1.00001f;
        clip[i] = v.x; clip[i + 1] = v.y; clip[i + 2] = v.z; clip[i + 3] = v.w;
        clip[i + 4] = __int_as_float((int)r2);
    }
}
extern "C" int probe(const void *gen, int blocks, float *cells, float *clip)
{
    k_probe<<<blocks, 32>>>((const double4_32a *)gen, cells, clip);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    d = tmp_path_factory.mktemp("vertex")
    src, lib = d / "probe.cu", d / "libprobe.so"
    src.write_text(PROBE)
    subprocess.run([BD.nvcc(), *BD.ARCH, "-O3", "-std=c++17", "--expt-relaxed-constexpr", "-diag-suppress", "1444",
                    "-Xcompiler", "-fPIC", "-shared", "-I", BD.CSRC, "-I", BD.INCLUDE, str(src), "-o", str(lib)],
                   check=True, capture_output=True)
    L = ctypes.CDLL(str(lib))
    L.probe.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p]
    return L.probe


@pytest.mark.parametrize("kind,scale", [("random", 1.0), ("lattice", 1.0), ("lattice", 2.0 ** -20), ("random", 2.0 ** 31)])
def test_same_vertex_and_bound(probe, kind, scale):
    """Neighbours of a random set, of a barely jittered lattice (nearly
    parallel and nearly co-spherical planes, exact solves among them), and at
    a scale where every vertex is solved exactly."""
    import torch
    rng = np.random.default_rng(1711)
    blocks = 400
    gen = np.zeros((blocks, 33, 4))
    if kind == "random":
        gen[:, :, :3] = rng.uniform(0.0, 1.0, (blocks, 33, 3))
    else:
        k = np.stack(np.meshgrid(*[np.arange(3.0)] * 3, indexing="ij"), -1).reshape(-1, 3) - 1.0
        near = k[np.argsort((k * k).sum(1), kind="stable")]
        gen[:, :27, :3] = near
        gen[:, 27:, :3] = 2.0 * near[1:7]
        gen[:, :, :3] += 1e-3 * rng.normal(size=(blocks, 33, 3))
        gen[:, :, :3] /= 64.0
    gen[:, :, :3] *= scale
    G = torch.tensor(gen.reshape(-1, 4), dtype=torch.float64, device="cuda")
    out = [torch.zeros(blocks * 32 * 64 * 5, dtype=torch.float32, device="cuda") for _ in range(2)]
    torch.cuda.synchronize()
    assert probe(G.data_ptr(), blocks, out[0].data_ptr(), out[1].data_ptr()) == 0
    a, b = (o.view(torch.int32).reshape(-1, 5) for o in out)
    formed = (out[1].reshape(-1, 5)[:, 3] > 0).sum().item()
    assert formed > 0.9 * blocks * 32 * 64
    bad = (a != b).any(dim=1)
    assert not bool(bad.any()), (int(bad.sum()), formed, out[0].reshape(-1, 5)[bad][:3], out[1].reshape(-1, 5)[bad][:3])
