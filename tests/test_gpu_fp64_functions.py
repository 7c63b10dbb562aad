"""The functions of the double-precision step (kf_fp64.cuh) on their own,
against extended precision (quadruple on AArch64), in units built with and
without -ftz=true.

Tolerances, U = 2^-53 (half an ulp of 1), from the operations of each function:
  from_float, to_float   exact, and rounded to nearest even, for every class
  rcp, sqrt              one rounding, the rest below 2^-10 of it
  rsqrt                  two roundings of half an ulp
  sincos                 the table entry's, the inner and the outer sum's
                         rounding (3 U of the result), and of |r| < 0.0123 the
                         entry's share, reduction 2 U, series 2.3 U, other
                         entry 1 U; relative where the entry is 0: reduction
                         2 U, series 1.3 U and its own rounding
  angle                  the sine and cosine handed in (6 U), the entries'
                         errors, the products' and the last sum's roundings;
                         relative to small angles: argument, series, sum
  sinc                   argument, reciprocal and product; its derivative's
                         numerator has the absolute errors of both terms
  wrap_phi               two roundings below pi, within a rounding of (-pi, pi]"""
import ctypes
import subprocess

import numpy as np
import pytest
import torch

from paper_2401_14221_gb300 import build as kbuild

pytestmark = pytest.mark.gpu
U = 2.0 ** -53
LD = np.longdouble
PI = LD("3.14159265358979323846264338327950288")

SOURCE = """
#include "kf_fp64.cuh"
namespace F = kf::f64;
__global__ void k(int f, int n, const double *a, const double *b, double *o0, double *o1) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double x = a[i], y = b[i];
  double r0 = 0.0, r1 = 0.0;
  if (f == 0) r0 = F::rcp(x);
  if (f == 1) r0 = F::rsqrt(x);
  if (f == 2) r0 = F::sqrt(x);
  if (f == 3) { const F::sc t = F::sincos(x); r0 = t.s; r1 = t.c; }
  if (f == 4) { const double q = 1.0 / ::hypot(x, y); r0 = F::angle(x, y, x * q, y * q); }
  if (f == 5) r0 = F::wrap_phi(x);
  if (f == 6) { const F::Sinc s = F::sinc(x, ::sin(x), ::cos(x)); r0 = s.S; r1 = s.dS; }
  o0[i] = r0;
  o1[i] = r1;
}
__global__ void conv(int n, const float *f, double *df, const double *d, float *fd) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  df[i] = F::from_float(f[i]);
  fd[i] = F::to_float(d[i]);
}
extern "C" int run(int f, int n, const double *a, const double *b, double *o0, double *o1) {
  k<<<(n + 127) / 128, 128>>>(f, n, a, b, o0, o1);
  return cudaDeviceSynchronize();
}
extern "C" int convert(int n, const float *f, double *df, const double *d, float *fd) {
  conv<<<(n + 127) / 128, 128>>>(n, f, df, d, fd);
  return cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module", params=[[], kbuild.FTZ_FLAGS], ids=["ieee", "ftz"])
def lib(request, tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tmp_path_factory.mktemp("fp64")
    (d / "f.cu").write_text(SOURCE)
    r = subprocess.run([kbuild._nvcc(), *kbuild.ARCH, *kbuild.NVCC_FLAGS, *request.param, "-shared",
                        "-cudart", "static", str(d / "f.cu"), "-o", str(d / "libf.so")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    torch.cuda.init()
    return ctypes.CDLL(str(d / "libf.so"))


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def call(lib, f, a, b=None):
    a = dev(a)
    b = a if b is None else dev(b)
    o0, o1 = torch.empty_like(a), torch.empty_like(a)
    torch.cuda.synchronize()
    p = [ctypes.c_void_p(t.data_ptr()) for t in (a, b, o0, o1)]
    assert lib.run(f, a.numel(), *p) == 0
    return o0.cpu().numpy().astype(LD), o1.cpu().numpy().astype(LD)


def ulp(x):
    return np.spacing(np.abs(x).astype(np.float64)).astype(LD)


def wide(n, lo, hi, seed):
    """Signs and exponents from 2^lo to 2^hi."""
    rng = np.random.default_rng(seed)
    return np.exp2(rng.uniform(lo, hi, n)) * rng.choice([-1.0, 1.0], n)


def test_conversions(lib):
    rng = np.random.default_rng(1)
    f = np.concatenate([rng.integers(0, 2 ** 32, 200000, dtype=np.uint32).view(np.float32),
                        np.arange(0, 70000, dtype=np.uint32).view(np.float32),
                        rng.integers(0, 2 ** 23, 50000, dtype=np.uint32).view(np.float32),
                        np.float32([0.0, -0.0, np.inf, -np.inf, np.nan, 2.0 ** -126, 2.0 ** -149])])
    with np.errstate(all="ignore"):
        near = f.astype(np.float64) * (1 + rng.integers(-4, 5, f.size) * 2.0 ** -25)  # ties and their sides
    d = np.where(rng.random(f.size) < 0.5, near, wide(f.size, -160, 130, 2))
    t = [dev(f), torch.empty(f.size, dtype=torch.float64, device="cuda"), dev(d),
         torch.empty(f.size, dtype=torch.float32, device="cuda")]
    torch.cuda.synchronize()
    assert lib.convert(f.size, *[ctypes.c_void_p(x.data_ptr()) for x in t]) == 0
    with np.errstate(all="ignore"):
        for got, want in ((t[1].cpu().numpy(), f.astype(np.float64)),
                          (t[3].cpu().numpy(), d.astype(np.float32))):
            assert np.array_equal(got, want, equal_nan=True)
            nan = np.isnan(want)
            assert np.array_equal(np.signbit(got)[~nan], np.signbit(want)[~nan])


@pytest.mark.parametrize("span", [(-8, 8), (-59, 59), (-140, 140)], ids=str)
def test_reciprocal_and_roots(lib, span):
    x = wide(200000, *span, 3)
    a = np.abs(x)
    for f, arg, want, tol in ((0, x, 1 / x.astype(LD), 0.501), (1, a, 1 / np.sqrt(a.astype(LD)), 1.001),
                              (2, a, np.sqrt(a.astype(LD)), 0.501)):
        err = np.abs(call(lib, f, arg)[0] - want) / ulp(want)
        assert err.max() <= tol, (f, float(err.max()))


def test_sine_and_cosine(lib):
    rng = np.random.default_rng(4)
    x = np.concatenate([rng.uniform(-64, 64, 300000), rng.uniform(-3.2, 3.2, 100000),
                        wide(100000, -60, -6.5, 5), np.arange(-2600, 2601) * (np.pi / 128)])
    s, c = call(lib, 3, x)
    for got, want in ((s, np.sin(x.astype(LD))), (c, np.cos(x.astype(LD)))):
        err = np.abs(got - want)
        assert np.all(err <= U * (3 * np.abs(want) + 6.4 * 0.0123))
    # pi/128 is reduced by as a double and a rest, which leaves `rest` a step
    rest = np.abs(PI / 128 - LD(0.02454369260617026) - LD(9.567553118338697e-19))
    k = np.arange(-40, 41) * (np.pi / 2)  # next to every zero of sin and cos
    x = np.concatenate([k * (1 + j * 2.0 ** -52) + d for j in range(-3, 4)
                        for d in (0.0, 1e-9, -1e-6, 1e-3, 0.01)])
    s, c = call(lib, 3, x)
    for got, want in ((s, np.sin(x.astype(LD))), (c, np.cos(x.astype(LD)))):
        small = np.abs(want) < 0.012
        step = np.abs(np.rint(x * (128 / np.pi))) * rest
        assert np.all((np.abs(got - want) <= 4.3 * U * np.abs(want) + step)[small])


@pytest.mark.parametrize("scale", [0, 90, -90], ids=str)
def test_angle(lib, scale):
    rng = np.random.default_rng(6)
    h = np.concatenate([rng.uniform(-np.pi, np.pi, 200000), wide(100000, -50, -6.5, 7)])
    r = np.exp2(rng.uniform(scale - 8, scale + 8, h.size))
    y, x = r * np.sin(h), r * np.cos(h)
    want = np.arctan2(y.astype(LD), x.astype(LD))
    err = np.abs(call(lib, 4, y, x)[0] - want)
    # the sine and cosine handed in: norm (2 ulp), reciprocal and product, 6 U
    assert np.all(err <= U * (6 + 2.1 + np.abs(want)))
    small = np.abs(want) < 0.012
    assert np.all(err[small] <= U * 8 * np.abs(want[small]))


@pytest.mark.parametrize("scale", [-125, -140, -300], ids=str)
def test_angle_of_tiny_operands(lib, scale):
    # below the range of a float, where the table angle cannot come from floats
    test_angle(lib, scale)


def test_sinc(lib):
    h = np.concatenate([wide(200000, -40, 1.6, 8), np.linspace(0.0499, 0.0501, 1001)])
    S, dS = call(lib, 6, h)
    H = h.astype(LD)
    tiny = np.abs(h) < 1e-3
    q = H * H
    wS = np.where(tiny, 1 - q / 6 * (1 - q / 20 * (1 - q / 42)), np.sin(H) / H)
    wd = np.where(tiny, -H / 3 * (1 - q / 10 * (1 - q / 28 * (1 - q / 54))), (np.cos(H) - wS) / H)
    assert np.all(np.abs(S - wS) <= U * (2 * 2 + 2) * np.abs(wS))
    quotient = np.abs(h) >= 0.05
    assert np.all(np.abs(dS - wd)[~quotient] <= U * 6 * np.abs(wd[~quotient]))
    assert np.all(np.abs(dS - wd)[quotient] <= (U * (10 / np.abs(H) + 3 * np.abs(wd)))[quotient])


def test_wrap(lib):
    rng = np.random.default_rng(9)
    edge = (2 * rng.integers(-1000, 1000, 20000) + 1) * np.pi
    a = np.concatenate([wide(100000, -20, 40, 10), edge + rng.uniform(-1e-6, 1e-6, 20000), edge])
    w = call(lib, 5, a)[0]
    # the azimuth of both edges is +-pi to the nearest doubles, one of them above pi
    assert np.all(np.abs(w) <= np.nextafter(np.pi, 4.0))
    A = a.astype(LD)
    n = np.rint((A - w) / (2 * PI))
    assert np.all(np.abs(A - w - n * 2 * PI) <= U * 2 * 3.15 + np.abs(n) * 2.0 ** -105)
