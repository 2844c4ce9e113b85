"""The integer contractions and the reciprocal / square root of the kernels on
the device, against exact sums of the same doubles: a small library built
around the headers (dg_fixed.cuh, dg_physics.cuh) exposes them one by one."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = r"""
#include "dg_fixed.cuh"
#include "dg_physics.cuh"
using namespace dgk;
__global__ void k_scalar(const double* a, double* r, double* s, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    r[i] = rcp(a[i]);
    s[i] = sqrt_hw(a[i]);
  }
}
// one block per field: [5][n^3] in, D_l of it out for l = 0..2
template <int n>
__global__ void k_grad(const double* in, double* out) {
  __shared__ double a[5 * n * n * n];
  for (int w = threadIdx.x; w < 5 * n * n * n; w += blockDim.x) a[w] = in[blockIdx.x * 5 * n * n * n + w];
  __syncthreads();
  fx_grad<n>(a, out + (int64_t)blockIdx.x * 15 * n * n * n);
}
extern "C" int scalar(const double* a, double* r, double* s, int64_t n) {
  k_scalar<<<256, 256>>>(a, r, s, n);
  return (int)cudaDeviceSynchronize();
}
template <int n>
int run(const double* in, double* out, int fields) {
  k_grad<n><<<fields, 96>>>(in, out);
  return (int)cudaDeviceSynchronize();
}
extern "C" int grad(int n, const double* in, double* out, int fields) {
  switch (n) {
    case 2: return run<2>(in, out, fields);
    case 3: return run<3>(in, out, fields);
    case 4: return run<4>(in, out, fields);
    case 5: return run<5>(in, out, fields);
    case 6: return run<6>(in, out, fields);
    default: return run<7>(in, out, fields);
  }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2511_08020_gb300 import build as b
    d = tmp_path_factory.mktemp("fixed")
    src, so = d / "t.cu", d / "t.so"
    src.write_text(CODE)
    subprocess.run([b.nvcc(), *b.ARCH, *b.FLAGS, "-I", b.CSRC, "-shared", "-o", str(so), str(src)], check=True,
                   capture_output=True)
    return ctypes.CDLL(str(so))


def p(t):
    return ctypes.c_void_p(t.data_ptr())


def test_reciprocal_and_root(lib):
    """Within 0.51 units of the last place of the exact value over the whole
    range, and the special values of the division and the root."""
    rng = np.random.Generator(np.random.PCG64(1))
    a = np.exp(rng.uniform(-700, 700, 20000)) * rng.uniform(1, 2, 20000)
    a = np.concatenate([a, rng.uniform(0.5, 4, 20000), 1 + np.arange(2000) * 2.0 ** -52])
    special = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, 1e-310, 1.7e308, -2.0, 2.2250738585072014e-308])
    x = torch.from_numpy(np.concatenate([a, special])).cuda()
    r, s = torch.empty_like(x), torch.empty_like(x)
    assert lib.scalar(p(x), p(r), p(s), ctypes.c_int64(x.numel())) == 0
    r, s = r.cpu().numpy(), s.cpu().numpy()
    from fractions import Fraction
    for k in range(0, len(a), 7):
        got, ref = Fraction(float(r[k])), 1 / Fraction(float(a[k]))
        assert abs(got - ref) <= Fraction(51, 100) * Fraction(float(np.spacing(1.0 / a[k])))
        # |s - sqrt(a)| <= 0.51 ulp: compare squares
        u = Fraction(51, 100) * Fraction(float(np.spacing(math.sqrt(a[k]))))
        g = Fraction(float(s[k]))
        assert (g - u) ** 2 <= Fraction(float(a[k])) <= (g + u) ** 2
    with np.errstate(all="ignore"):
        np.testing.assert_array_equal(r[len(a):], 1.0 / special)
        np.testing.assert_array_equal(s[len(a):], np.sqrt(special))


@pytest.mark.parametrize("n", range(2, 8))
def test_contraction(lib, n):
    """D_l of fields of widely differing scales against the sums of the same
    products without rounding error: within 16 x 2^-53 of the row's sum of
    |coefficient| times the line's largest value (the reference's matrix, built
    in double, carries a few units itself) plus one unit of its own last place;
    exact zeros, and NaN for lines that hold a non-finite value."""
    from numpy.polynomial import legendre
    rng = np.random.Generator(np.random.PCG64(n))
    x = legendre.leggauss(n)[0]
    D = np.empty((n, n))                                   # D[i][m] = l'_m(x_i) (barycentric)
    lam = np.array([1 / np.prod(x[i] - np.delete(x, i)) for i in range(n)])
    for i in range(n):
        for m in range(n):
            if i != m:
                D[i, m] = lam[m] / lam[i] / (x[i] - x[m])
        D[i, i] = -sum(D[i, m] for m in range(n) if m != i)
    F = 8
    a = rng.uniform(-1, 1, size=(F, 5, n, n, n))
    a[1] *= 1e-200
    a[2] *= 1e250
    a[3] *= 10.0 ** rng.uniform(-12, 3, size=a[3].shape)   # mixed magnitudes within a line
    a[4] = 0.0
    a[5] = 180.0 + 1e-9 * a[5]                             # a constant but for its last digits
    a[6, 2, 0, 0, n - 1] = np.nan
    a[6, 3, 1, 1, 0] = np.inf
    a[7] = np.where(rng.uniform(size=a[7].shape) < 0.5, -0.0, 1e-300 * a[7])
    t = torch.from_numpy(a).cuda()
    out = torch.empty((F, 3, 5, n, n, n), dtype=torch.float64, device="cuda")
    assert lib.grad(n, p(t), p(out), F) == 0
    out = out.cpu().numpy()
    for l in range(3):
        got = np.moveaxis(out[:, l], 2 + l, -1)
        lines = np.moveaxis(a, 2 + l, -1)
        bad = ~np.isfinite(lines).all(axis=-1)
        assert np.isnan(got[bad]).all() and np.isfinite(got[~bad]).all()
        # the reference: products split exactly by math.fsum's exact summation of
        # the double products; D itself carries a few ulps
        ref = np.zeros_like(got)
        bound = np.zeros_like(got)
        for i in range(n):
            big = np.abs(np.where(np.isfinite(lines), lines, 0)).max(axis=-1)
            ref[..., i] = np.apply_along_axis(lambda v: math.fsum(D[i] * v), -1, np.where(bad[..., None], 0, lines))
            bound[..., i] = np.abs(D[i]).sum() * big
        err = np.abs(got - ref)[~bad]
        tol = (16 * 2.0 ** -53 * bound + np.spacing(np.abs(ref)))[~bad]
        assert (err <= tol + 1e-307).all(), (l, (err / (tol + 1e-307)).max())
    assert (out[4] == 0).all()
