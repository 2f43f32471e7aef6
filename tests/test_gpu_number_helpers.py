"""The library's own roots and conversions (pair_physics.cuh, common.cuh) by
themselves: the FP64 square root and its reciprocal within one unit in the last
place of the exact values over all normal numbers, the conversions on the
integer ALU bit for bit those of the hardware, ties, subnormal numbers,
infinities and overflow among them."""
import ctypes
import subprocess

import numpy as np
import pytest
import torch

from paper_2411_13992_gb300 import _build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "pair_physics.cuh"
using namespace sphtv;
__global__ void k_roots(int n, const double* x, double* s, double* r)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    s[i] = sqrt_pos(x[i]);
    r[i] = rsqrt_pos(x[i]);
}
__global__ void k_conversions(int n, const double* x, float* f, float* f_hw, double* half, double* half_hw)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    f[i] = d2f_rn(x[i]);
    f_hw[i] = __double2float_rn(x[i]);
    half[i] = half_exact(x[i]);
    half_hw[i] = 0.5 * x[i];
}
__global__ void k_widen(int n, const float* x, double* d, double* d_hw)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    d[i] = f2d_exact(x[i]);
    d_hw[i] = (double)x[i];
}
extern "C" __attribute__((visibility("default"))) int roots(int n, const double* x, double* s, double* r)
{
    k_roots<<<(n + 255) / 256, 256>>>(n, x, s, r);
    return (int)cudaDeviceSynchronize();
}
extern "C" __attribute__((visibility("default"))) int conversions(int n, const double* x, float* f, float* f_hw,
                                                                  double* half, double* half_hw)
{
    k_conversions<<<(n + 255) / 256, 256>>>(n, x, f, f_hw, half, half_hw);
    return (int)cudaDeviceSynchronize();
}
extern "C" __attribute__((visibility("default"))) int widen(int n, const float* x, double* d, double* d_hw)
{
    k_widen<<<(n + 255) / 256, 256>>>(n, x, d, d_hw);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    assert torch.cuda.is_available()
    d = tmp_path_factory.mktemp("helpers")
    (d / "helpers.cu").write_text(SOURCE)
    so = d / "helpers.so"
    subprocess.run([_build.nvcc(), *_build.ARCH, *_build.NVCC_FLAGS, "-shared", "-cudart", "static",
                    str(d / "helpers.cu"), "-o", str(so)], check=True, capture_output=True)
    return ctypes.CDLL(str(so))


def _call(f, x, *outs):
    args = [ctypes.c_int(x.numel())] + [ctypes.c_void_p(t.data_ptr()) for t in (x, *outs)]
    torch.cuda.synchronize()
    assert f(*args) == 0


def _doubles(exponents, rng, per_exponent):
    """Numbers of the given binary exponents: fractions at and beside both ends
    of the binade, with one bit set, and random ones."""
    ends = np.array([0, 1, 2, (1 << 52) - 1, (1 << 52) - 2, 1 << 51, (1 << 51) - 1, (1 << 51) + 1], np.uint64)
    ones = np.uint64(1) << np.arange(52, dtype=np.uint64)
    out = []
    for e in exponents:
        frac = np.concatenate([ends, ones, rng.integers(0, 1 << 52, per_exponent, dtype=np.uint64)])
        out.append((np.uint64(e + 1023) << np.uint64(52)) | frac)
    return np.concatenate(out).view(np.float64)


def test_roots_within_one_unit_in_the_last_place(lib):
    rng = np.random.default_rng(1)
    x = np.concatenate([_doubles(range(-1022, 1024), rng, 40), _doubles(range(-30, 10), rng, 20000)])
    xd = torch.from_numpy(x).cuda()
    s, r = torch.empty_like(xd), torch.empty_like(xd)
    _call(lib.roots, xd, s, r)
    wide = np.longdouble(x)
    for got, exact in ((s, np.sqrt(wide)), (r, 1 / np.sqrt(wide))):
        got = got.cpu().numpy()
        ulp = np.spacing(exact.astype(np.float64))
        err = np.abs((np.longdouble(got) - exact) / ulp)
        print("largest error %.4f ulp" % float(err.max()))
        assert np.isfinite(got).all() and err.max() < 1.0


def test_narrowing_and_halving_are_the_hardware_s(lib):
    rng = np.random.default_rng(2)
    x = _doubles(list(range(-1022, -150, 31)) + list(range(-152, 131)) + list(range(131, 1024, 31)), rng, 300)
    # ties and their neighbours at every kept bit of a float's last place
    keep = rng.integers(0, 1 << 23, 4000, dtype=np.uint64) << np.uint64(29)
    exps = (rng.integers(-130, 129, 4000) + 1023).astype(np.uint64) << np.uint64(52)
    ties = np.concatenate([(exps | keep | np.uint64(1 << 28)) + np.uint64(d) for d in (0, 1)] +
                          [(exps | keep | np.uint64(1 << 28)) - np.uint64(1)]).view(np.float64)
    top = np.float64(np.finfo(np.float32).max)
    edge = np.array([0.0, np.inf, np.nan, 5e-324, 2.0 ** -1022, 2.0 ** -1021, np.nextafter(2.0 ** -1021, 0), 2.0 ** -126,
                     np.nextafter(2.0 ** -126, 0), 2.0 ** -149, 2.0 ** -150, top, top + 2.0 ** 102, top + 2.0 ** 103,
                     np.finfo(np.float64).max])
    x = np.concatenate([x, ties, edge])
    x = np.concatenate([x, -x])
    xd = torch.from_numpy(x).cuda()
    f, fh = (torch.empty(len(x), dtype=torch.float32, device="cuda") for _ in range(2))
    h, hh = torch.empty_like(xd), torch.empty_like(xd)
    _call(lib.conversions, xd, f, fh, h, hh)
    assert torch.equal(f.view(torch.int32), fh.view(torch.int32))
    assert torch.equal(h.view(torch.int64), hh.view(torch.int64))


def test_widening_is_the_hardware_s(lib):
    rng = np.random.default_rng(3)
    bits = np.concatenate([(np.uint32(e) << np.uint32(23)) | np.concatenate(
        [np.array([0, 1, 2, (1 << 23) - 1, 1 << 22], np.uint32), np.uint32(1) << np.arange(23, dtype=np.uint32),
         rng.integers(0, 1 << 23, 200, dtype=np.uint32)]) for e in range(0, 255)] + [np.array([0x7f800000], np.uint32)])
    bits = np.concatenate([bits, bits | np.uint32(1 << 31)])
    xd = torch.from_numpy(bits.view(np.float32)).cuda()
    d, dh = (torch.empty(len(bits), dtype=torch.float64, device="cuda") for _ in range(2))
    _call(lib.widen, xd, d, dh)
    assert torch.equal(d.view(torch.int64), dh.view(torch.int64))
