"""The integer contractions of the element kernels (dg_fixed.cuh) compiled for
the host: one lane per block, so every loop over lanes runs in order and the
barriers do nothing.  Arithmetic and indexing are those of the device build."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2511_08020_gb300", "csrc")
CODE = r"""
#include <cuda_runtime.h>
#include <stdint.h>
#include <cmath>
#include <cstring>
#undef __shared__
#undef __constant__
#define __shared__ static
#define __constant__ static const
struct One { unsigned x; };
static One lane0 = {0}, lanes = {1};
#define threadIdx lane0
#define blockDim lanes
static inline int min(int a, int b) { return a < b ? a : b; }
static inline int max(int a, int b) { return a > b ? a : b; }
static inline unsigned min(unsigned a, unsigned b) { return a < b ? a : b; }
static inline unsigned max(unsigned a, unsigned b) { return a > b ? a : b; }
template <class T> static inline T bits(double x) { T t; memcpy(&t, &x, 8); return t; }
static inline long long __double_as_longlong(double x) { return bits<long long>(x); }
static inline double __longlong_as_double(long long x) { double d; memcpy(&d, &x, 8); return d; }
static inline int __double2hiint(double x) { return (int)(bits<uint64_t>(x) >> 32); }
static inline int __double2loint(double x) { return (int)bits<uint64_t>(x); }
static inline double __hiloint2double(int h, int l) { return __longlong_as_double((long long)(((uint64_t)(unsigned)h << 32) | (unsigned)l)); }
static inline unsigned __funnelshift_r(unsigned lo, unsigned hi, unsigned s) { return (unsigned)((((uint64_t)hi << 32) | lo) >> (s & 31)); }
static inline unsigned __funnelshift_l(unsigned lo, unsigned hi, unsigned s) { return (unsigned)(((((uint64_t)hi << 32) | lo) << (s & 31)) >> 32); }
static inline int __clz(int x) { return x ? __builtin_clz((unsigned)x) : 32; }
template <class T> static inline T __ldg(const T* p) { return *p; }
static inline void __syncthreads() {}
static inline int __syncthreads_or(int x) { return x; }
#include "dg_fixed.cuh"
#include "dg_host.h"
using namespace dgk;
namespace {
struct Setup {
  dgh::Tables tb;
  Ctx c{};
  const TypeTab& T;
  static dgh::Tables make(int type, int N) { dgh::Tables t; std::string e; t.add(type, N, &e); return t; }
  Setup(int type, int N) : tb(make(type, N)), T(tb.tabs[0]) {
    c.dpool = tb.dpool.data();
    c.ipool = tb.ipool.data();
    c.fpool = reinterpret_cast<const int2*>(tb.fpool.data());
  }
};
template <int n> void dsum(const double* G, unsigned dirs, double* out) {
  constexpr int m = 5 * n * n * n;
  double g[3 * m];
  memcpy(g, G, sizeof(g));
  // in place of G_2, as the element kernels call it, when that direction is the first
  double tmp[m];
  fx_dsum<n>([&](int l, int v, int q) { return g[(5 * l + v) * n * n * n + q]; }, dirs, (dirs & 4u) ? g + 2 * m : tmp, out);
}
template <int n> void lift(int type, const double* H, const double* F, int neg, double* out) {
  constexpr int m = 5 * n * n * n;
  Setup s(type, n - 1);
  double A[m];
  fx_lift<n>(s.T, [&](int o) { return H[o]; }, F, neg ? 0x80000000u : 0u, A, [&](int o, double x) { out[o] = x; });
}
template <int n> int lift_modal(int type, const double* H, const double* F, int neg, int stage, double* out) {
  constexpr int m = 5 * n * n * n, g = 15 * n * n * n > 30 * n * n ? 15 * n * n * n : 30 * n * n;
  Setup s(type, n - 1);
  double A[m], G[g];
  auto fH = [&](int o) { return H[o]; };
  auto fF = [&](int lf, int v, int p) { return F[(lf * 5 + v) * n * n + p]; };
  if (stage) fx_lift_to_modal<n, true>(s.c, s.T, fH, fF, neg ? 0x80000000u : 0u, A, G, A);
  else fx_lift_to_modal<n, false>(s.c, s.T, fH, fF, neg ? 0x80000000u : 0u, A, G, G + m);
  memcpy(out, stage ? A : G + m, 5 * s.T.nM * sizeof(double));
  return s.T.nM;
}
template <int n, bool IEEE> int nodal(int type, const double* Q, double* out, double* tr) {
  constexpr int n2 = n * n, m = 5 * n * n2;
  Setup s(type, n - 1);
  double A[m], B[m];
  memcpy(B, Q, 5 * s.T.nM * sizeof(double));
  fx_to_nodal<n, !IEEE, IEEE>(s.c, s.T, B, A, B, [&](int lf, int v, int p, double x) { tr[(lf * 5 + v) * n2 + p] = x; });
  memcpy(out, A, sizeof(A));
  return s.T.nM;
}
template <int n, bool IEEE> int modal(int type, const double* U, double* out) {
  constexpr int m = 5 * n * n * n;
  Setup s(type, n - 1);
  double A[m], B[m];
  memcpy(A, U, sizeof(A));
  fx_to_modal<n, IEEE>(s.T, s.c, A, B, B);
  memcpy(out, B, 5 * s.T.nM * sizeof(double));
  return s.T.nM;
}
template <int n> void grad(const double* U, double* out) { fx_grad<n>(U, out); }
}  // namespace
#define EACH(n, f) (n == 2 ? f<2> : n == 3 ? f<3> : n == 4 ? f<4> : n == 5 ? f<5> : n == 6 ? f<6> : f<7>)
#define EACH2(n, f, b) (n == 2 ? f<2, b> : n == 3 ? f<3, b> : n == 4 ? f<4, b> : n == 5 ? f<5, b> : n == 6 ? f<6, b> : f<7, b>)
extern "C" {
void t_dsum(int n, const double* G, unsigned dirs, double* out) { EACH(n, dsum)(G, dirs, out); }
void t_lift(int n, int type, const double* H, const double* F, int neg, double* out) { EACH(n, lift)(type, H, F, neg, out); }
int t_lift_modal(int n, int type, const double* H, const double* F, int neg, int stage, double* out) {
  return EACH(n, lift_modal)(type, H, F, neg, stage, out);
}
int t_nodal(int n, int type, int ieee, const double* Q, double* out, double* tr) {
  return ieee ? EACH2(n, nodal, true)(type, Q, out, tr) : EACH2(n, nodal, false)(type, Q, out, tr);
}
int t_modal(int n, int type, int ieee, const double* U, double* out) {
  return ieee ? EACH2(n, modal, true)(type, U, out) : EACH2(n, modal, false)(type, U, out);
}
void t_dense(int nM, const double* Md, const double* r, double* out) {
  dense_product(Md, r, nM, [&](int a, const double* acc) {
    for (int v = 0; v < 5; ++v) out[v * nM + a] = acc[v];
  });
}
void t_grad(int n, const double* U, double* out) { EACH(n, grad)(U, out); }
// a hexahedron's modal coefficients to its storage and back, as dg_set_state and dg_get_state do
int t_storage(int n, const double* Q, double* out) {
  Setup s(HEX, n - 1);
  const double* sq = s.c.dpool + s.T.sqw;
  const int nQ = n * n * n;
  double U[5 * 343];
  EACH2(n, nodal, true)(HEX, Q, U, nullptr);
  for (int o = 0; o < 5 * nQ; ++o) U[o] = U[o] * sq[o % nQ] * sq[2 * nQ + o % nQ];
  return EACH2(n, modal, true)(HEX, U, out);
}
// largest 64-bit sum of the ragged passes and of the lift over its limit 2^63,
// for operands h 2^31 + l with |h| <= 2^30 (2^31 in the lift at a node), 0 <= l < 2^31
double t_bounds(int n, int type) {
  Setup s(type, n - 1);
  const TypeTab& T = s.T;
  const int* ip = s.c.ipool;
  double worst = 0.0;
  auto sum = [&](int off, int cnt, int stride, int hb, double times) {
    double mid = 0.0, top = 0.0;
    for (int k = 0; k < cnt; ++k) {
      const dgk::FixPair c = s.tb.fpool[off + k * stride];
      mid += ldexp(fabs((double)c.y), hb) + ldexp(fabs((double)c.x), 31);
      top += ldexp(fabs((double)c.x), hb);
    }
    worst = fmax(worst, ldexp(fmax(times * mid + ldexp(1.0, 30), times * top + ldexp(1.0, 32)), -63));
  };
  for (int p = 0; p < n; ++p) {
    const int off = T.B + ip[T.p_boff + p], len = ip[T.p_blen + p];
    for (int k = 0; k < n; ++k) sum(off + k, len, n, 30, 1.0);
    for (int r = 0; r < len; ++r) sum(off + r * n, n, 1, 30, 1.0);
  }
  for (int col = 0; col < T.ncols; ++col) {
    const int off = T.C + ip[T.col_coff + col], len = ip[T.col_len + col];
    for (int k = 0; k < n; ++k) sum(off + k, len, n, 30, 1.0);
    for (int r = 0; r < len; ++r) sum(off + r * n, n, 1, 30, 1.0);
  }
  for (int i = 0; i < n; ++i) {
    sum(T.ext + i, 2, n, 30, 3.0);
    sum(T.ext + i, 2, n, 31, 1.0);
  }
  return worst;
}
// nodes, Lagrange end values, and the factors of the basis at the nodes
int t_tables(int n, int type, double* A, double* V, double* ext, int* face) {
  Setup s(type, n - 1);
  const TypeTab& T = s.T;
  const double* dp = s.c.dpool;
  const int* ip = s.c.ipool;
  for (int k = 0; k < n * n; ++k) A[k] = dp[T.A + k];
  for (int k = 0; k < 2 * n; ++k) ext[k] = dp[T.ext + k];
  for (int k = 0; k < 6; ++k) face[k] = T.face_of[k];
  for (int mode = 0; mode < T.nM; ++mode) {
    const int col = ip[T.mode_col + mode], t = mode - ip[T.col_moff + col], p = ip[T.col_p + col], q = col - ip[T.p_cbase + p];
    for (int i = 0; i < n; ++i)
      for (int j = 0; j < n; ++j)
        for (int k = 0; k < n; ++k)
          V[((i * n + j) * n + k) * T.nM + mode] = dp[T.A + p * n + i] * dp[T.B + ip[T.p_boff + p] + q * n + j] *
                                                   dp[T.C + ip[T.col_coff + col] + t * n + k];
  }
  return T.nM;
}
}
"""


def build(tmp):
    src, so = os.path.join(tmp, "fx.cpp"), os.path.join(tmp, "fx.so")
    with open(src, "w") as f:
        f.write(CODE)
    from paper_2511_08020_gb300 import build as b
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(b.nvcc()))), "include")
    r = subprocess.run(["g++", "-O1", "-std=c++17", "-fPIC", "-shared", "-w", "-fsanitize=shift-exponent,bounds,signed-integer-overflow",
                        "-fsanitize-undefined-trap-on-error", "-I", CSRC, "-isystem", inc,
                        "-I", os.path.join(ROOT, "include"), "-o", so, src, os.path.join(CSRC, "dg_host.cpp"), "-lpthread"],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(so)


def nodes(n):
    """Gauss-Legendre nodes, D[i][m] = l'_m(x_i) and E[end][m] = l_m(-+1) in extended precision."""
    x = np.polynomial.legendre.leggauss(n)[0].astype(np.longdouble)
    for _ in range(3):
        p0, p1 = np.ones_like(x), x
        for k in range(2, n + 1):
            p0, p1 = p1, ((2 * k - 1) * x * p1 - (k - 1) * p0) / k
        x = x - p1 * (x * x - 1) / (n * (x * p1 - p0))
    x = (x - x[::-1]) / 2
    lam = np.array([1 / np.prod([x[i] - x[j] for j in range(n) if j != i]) for i in range(n)])
    D = np.zeros((n, n), np.longdouble)
    for i in range(n):
        for m in range(n):
            if i != m:
                D[i, m] = lam[m] / lam[i] / (x[i] - x[m])
        D[i, i] = 0 if 2 * i + 1 == n else -D[i].sum()
    E = np.array([[np.prod([(y - x[k]) / (x[m] - x[k]) for k in range(n) if k != m]) for m in range(n)] for y in (-1, 1)])
    return x, D, E


def tables(fx, n, etype):
    """V [points][modes] and the local faces at the ends of the collapsed coordinates."""
    A, V, ext, face = np.empty(n * n), np.zeros(n ** 6), np.empty(2 * n), np.empty(6, np.int32)
    nM = fx.t_tables(n, etype, ptr(A), ptr(V), ptr(ext), ptr(face))
    return V[:n ** 3 * nM].reshape(n ** 3, nM), face


def ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


@pytest.fixture(scope="session")
def fx(tmp_path_factory):
    return build(str(tmp_path_factory.mktemp("fx")))
