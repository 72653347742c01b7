"""The short FP64 sequences of mm_fp64.cuh against CUDA's operations and exact
rational arithmetic.

Bounds.  The seeds (rcp/rsqrt.approx.ftz.f64) read and give upper words, 20
bits of mantissa, so their relative error is taken as at most 2^-19; an ulp is
at least 2^-53 of its number.
* rcp64: e <= 2^-19, the series stops short of e^3 <= 2^-57, 1/16 ulp, then
  one rounding: 0.5 + 1/16 ulp.
* rsqrt64: e = 1 - x y^2 <= 2^-18, the series stops short of 5/16 e^3,
  5/32 ulp: 0.5 + 5/32 ulp.
* sqrt64, div64: the residual step multiplies a correction of a few ulp by the
  seed or a reciprocal within 2^-19: 0.5 + 2^-16 ulp.
2^-16 is added to each for the roundings inside the corrections (2^-19 of an
ulp).  Outside the range of the seeds every function is CUDA's operation, bit
for bit: zeros, subnormals, infinities and NaN, with their signs."""
import ctypes
import math
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_1707_05333_gb300 import build as BD

pytestmark = pytest.mark.gpu

PROBE = r"""
#include <cuda_runtime.h>
#include "mm_fp64.cuh"
using namespace mm;
__global__ void k_probe(const double *a, const double *b, long n, double *out)
{
    const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    out[i] = rcp64(a[i]);
    out[n + i] = rsqrt64(a[i]);
    out[2 * n + i] = sqrt64(a[i]);
    out[3 * n + i] = div64(a[i], b[i]);
    out[4 * n + i] = 1.0 / a[i];
    out[5 * n + i] = rsqrt(a[i]);
    out[6 * n + i] = sqrt(a[i]);
    out[7 * n + i] = a[i] / b[i];
}
extern "C" int probe(const double *a, const double *b, long n, double *out)
{
    k_probe<<<(unsigned)((n + 127) / 128), 128>>>(a, b, n, out);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    import torch
    d = tmp_path_factory.mktemp("fp64")
    src, lib = d / "probe.cu", d / "libprobe.so"
    src.write_text(PROBE)
    subprocess.run([BD.nvcc(), *BD.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-I", BD.CSRC,
                    str(src), "-o", str(lib)], check=True, capture_output=True)
    L = ctypes.CDLL(str(lib))
    L.probe.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_long, ctypes.c_void_p]

    def run(a, b):
        A, B = (torch.tensor(np.asarray(x, dtype=np.float64), device="cuda") for x in (a, b))
        out = torch.empty((8, len(A)), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert L.probe(A.data_ptr(), B.data_ptr(), len(A), out.data_ptr()) == 0
        o = out.cpu().numpy()
        return dict(zip(("rcp", "rsqrt", "sqrt", "div"), o[:4])), dict(zip(("rcp", "rsqrt", "sqrt", "div"), o[4:]))

    return run


def ulp(x):
    return Fraction(math.ulp(float(x)))


def test_inside_the_range(probe):
    """Random mantissas (and those beside powers of two) at exponents over the
    whole range the sequences take."""
    rng = np.random.default_rng(1707)
    m = rng.uniform(1.0, 2.0, 12000)
    m[:600] = np.repeat([1.0, np.nextafter(1.0, 2.0), np.nextafter(2.0, 1.0), 1.5, math.sqrt(2.0), 4.0 / 3.0], 100)
    e = rng.integers(-1000, 1000, len(m))
    x = np.ldexp(m, e)
    # a / b: half with quotients near one, half anywhere the result is normal
    mb, eb = rng.uniform(1.0, 2.0, len(m)), np.clip(e + rng.integers(-3, 4, len(m)), -1000, 999)
    far = rng.random(len(m)) < 0.5
    eb[far] = rng.integers(-1000, 1000, far.sum())
    eb = np.clip(eb, e - 1015, e + 1015)
    b = np.ldexp(mb, eb) * rng.choice([-1.0, 1.0], len(m))
    got, lib = probe(x, b)
    small = Fraction(1, 2 ** 16)
    bound = {"rcp": Fraction(1, 2) + Fraction(1, 16) + small, "rsqrt": Fraction(1, 2) + Fraction(5, 32) + small,
             "sqrt": Fraction(1, 2) + small, "div": Fraction(1, 2) + small}
    for k in range(len(x)):
        X, B = Fraction(float(x[k])), Fraction(float(b[k]))
        for name in bound:
            r = Fraction(float(got[name][k]))
            d = bound[name] * ulp(got[name][k])
            lo, hi = r - d, r + d
            if name == "rcp":
                ok = lo * X <= 1 <= hi * X
            elif name == "rsqrt":
                ok = lo * lo * X <= 1 <= hi * hi * X
            elif name == "sqrt":
                ok = lo * lo <= X <= hi * hi
            else:
                ok = min(lo * B, hi * B) <= X <= max(lo * B, hi * B)
            assert ok, (name, float(x[k]).hex(), float(b[k]).hex(), float(got[name][k]).hex())
    for name in bound:  # and within an ulp of CUDA's
        assert np.all(np.abs(got[name] - lib[name]) <= np.spacing(np.abs(lib[name]))), name


def same_bits(g, r):
    return np.where(np.isnan(r), np.isnan(g), g.view(np.int64) == r.view(np.int64))


def test_ends_of_the_range(probe):
    """Zeros, subnormals, the largest and smallest normal numbers, infinities
    and NaN, as arguments, dividends and divisors: CUDA's result bit for bit."""
    rng = np.random.default_rng(1708)
    tiny, big = np.finfo(float).tiny, np.finfo(float).max
    ends = [0.0, 5e-324, 1e-320, tiny, np.nextafter(tiny, 0.0), 2.0 ** -1001, np.nextafter(2.0 ** -1000, 0.0),
            2.0 ** 1000, 2.0 ** 1001, 2.0 ** 1022, big, np.inf, np.nan]
    ends += list(np.ldexp(rng.uniform(1.0, 2.0, 40), rng.integers(-1074, -1000, 40)))
    ends += list(np.ldexp(rng.uniform(1.0, 2.0, 40), rng.integers(1000, 1024, 40)))
    ends = np.array(ends + [-v for v in ends])
    got, lib = probe(ends, np.ones_like(ends))
    for name in ("rcp", "rsqrt", "sqrt"):
        ok = same_bits(got[name], lib[name])
        assert np.all(ok), (name, ends[~ok][:4], got[name][~ok][:4], lib[name][~ok][:4])
    # every pair of two ends, and of an end with an ordinary number on either side
    plain = np.array([1.0, -1.0, 3.0, -0.7, 2.0 ** 300, -(2.0 ** -300), 1e100])
    pool = np.concatenate([ends, plain])
    a, b = (v.ravel() for v in np.meshgrid(pool, pool, indexing="ij"))
    edge = ~(np.isin(a, plain) & np.isin(b, plain))
    got, lib = probe(a[edge], b[edge])
    ok = same_bits(got["div"], lib["div"])
    assert np.all(ok), [(a[edge][k], b[edge][k], got["div"][k], lib["div"][k]) for k in np.flatnonzero(~ok)[:6]]
