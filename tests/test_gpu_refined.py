"""The FP64 roots, quotients and reciprocals refined from the hardware's float ones (peskin.cuh,
fft_lines.cuh), against IEEE square roots and divisions: over random arguments, at both ends of the
range they take (beyond it the ordinary operations follow) and at significands of few and of all
bits.  The kernel below is compiled from those headers.

Each value before its last rounding is good to 2^-85 or better, so one random argument in 2^32 may
round to the other neighbour: none or one of the 2^22 here, and by one ulp.  Arguments next to powers
of two have roots and quotients within 2^-100 of a midpoint, which may go either way: one ulp.
"""
import ctypes
import subprocess

import numpy as np
import pytest

import oracle
from helpers import rel_l2, to_np

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("CUDA device required", allow_module_level=True)

import paper_1407_5600_gb300 as mb  # noqa: E402
from paper_1407_5600_gb300 import build as cuda_build  # noqa: E402
from paper_1407_5600_gb300 import workloads as wl  # noqa: E402

SOURCE = """
#include "fft_lines.cuh"
#include "peskin.cuh"
__global__ void k(long n, const double* a, const double* x, double* root, double* len, double* quo, double* rec)
{
    const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    root[i] = mbk::peskin_sqrt(0.25 + 0.75 * (a[i] - floor(a[i])));
    const mbk::Length l(a[i]);
    len[i] = l.len;
    quo[i] = l.divide(x[i]);
    rec[i] = mbk::recip(a[i]);
}
extern "C" int run(long n, const double* a, const double* x, double* root, double* len, double* quo, double* rec)
{
    k<<<(unsigned)((n + 255) / 256), 256>>>(n, a, x, root, len, quo, rec);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def refined(tmp_path_factory):
    d = tmp_path_factory.mktemp("refined")
    (d / "k.cu").write_text(SOURCE)
    subprocess.run([cuda_build.nvcc(), *cuda_build.ARCH, "-O3", "-std=c++17", "-shared", "-cudart", "shared",
                    "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr", "-I", cuda_build.CSRC, "-o", str(d / "k.so"),
                    str(d / "k.cu")], check=True)
    lib = ctypes.CDLL(str(d / "k.so"))

    def call(a, x):
        a, x = (torch.as_tensor(t, device="cuda") for t in (a, x))
        out = [torch.empty_like(a) for _ in range(4)]
        torch.cuda.synchronize()
        assert lib.run(ctypes.c_long(len(a)), *(ctypes.c_void_p(t.data_ptr()) for t in (a, x, *out))) == 0
        return [t.cpu().numpy() for t in out]

    return call


def _agree(got, want, most):
    """At most `most` of the values differ, by one ulp."""
    same = (got == want) | (np.isnan(got) & np.isnan(want))
    off = np.abs(got[~same].view(np.int64) - want[~same].view(np.int64))
    assert len(off) <= most and np.all(off <= 1), (len(off), got[~same][:3], want[~same][:3])


def _check(refined, a, x, most):
    root, length, quo, rec = refined(a, x)
    with np.errstate(all="ignore"):
        t = 0.25 + 0.75 * (a - np.floor(a))
        ok = np.isfinite(t)
        _agree(length, np.sqrt(a), most)
        _agree(quo, x / length, most)
        _agree(rec, 1.0 / a, most)
        assert np.all(np.abs(root[ok] / np.sqrt(t[ok]) - 1.0) <= 2.0 ** -51)      # t itself may be fused


@pytest.mark.parametrize("lo,hi", [(-3, 3), (-30, 30), (-126, 126), (-300, 300)])
def test_refined_operations(refined, lo, hi):
    rng = np.random.default_rng(hi)
    n = 1 << 22
    a = np.ldexp(1.0 + rng.random(n), rng.integers(lo, hi, n))
    _check(refined, a, rng.normal(size=n), 1)


def test_refined_operations_at_their_limits(refined):
    one = np.float64(1.0)
    m = [one, np.nextafter(one, 2), np.nextafter(np.float64(2), 1), 1.5, 1.0 + 2.0 ** -23, 2.0 - 2.0 ** -23,
         1.0 + 2.0 ** -24, 2.0 - 2.0 ** -24, 1.0 + 2.0 ** -26, 1.999999]
    e = [-1074, -1022, -300, -149, -128, -127, -126, -125, -1, 0, 1, 63, 125, 126, 127, 128, 300, 1023]
    a = np.array([np.ldexp(x, k) for x in m for k in e] + [0.0, np.inf, np.nan])
    rng = np.random.default_rng(1)
    for x in (np.ones_like(a), rng.normal(size=len(a)), -np.ldexp(1.0, rng.integers(-60, 60, len(a)))):
        _check(refined, a, x, len(a))


@pytest.mark.parametrize("rho", [1e38, 8.6e37, 1.6e38, 1.1e-38])
def test_fluid_update_where_the_divisor_leaves_the_float_range(rho):
    """rho/dt about 2^126 and 2^-126, five FP64 passes."""
    n, kw = (4, 8, 256), dict(h=0.8, rho=rho, eta=0.1 * rho, dt=1.0)
    v = wl.random_field(n[::-1], 5)
    with mb.Multiblob(mb.GridDesc(*n, precision=1, **kw)) as sim:
        got = to_np(sim.fluid_update(v))[0]
    g = oracle.Grid(*n, **kw)
    assert rel_l2(got, oracle.fluid_update(g, v, g.zeros())) < 1e-13
