// Element kernels of the modal DG hot path, compiled once per number of points
// per direction (DG_N = N + 1 = 2..7): every loop bound, buffer size and index
// division is a constant, and a launch carries the registers of its own degree
// only.  Each degree is built in three parts side by side: the stage phases
// (DG_PART 0), the Navier-Stokes volume phase, one-shot maps and stage mass
// solves (1), the adjoint phases (2).  See dg_kernels.cuh for the phase layout.
#include <algorithm>

#if DG_PART == 1
#define DG_UNROLL 1
#endif
#include "dg_fixed.cuh"
#include "dg_physics.cuh"

#if !defined(DG_N) || !defined(DG_PART)
#error "DG_N (points per direction) and DG_PART must be defined"
#endif

namespace dgk {

namespace {

constexpr int kn = DG_N, kn2 = kn * kn, knQ = kn2 * kn;
// bufG of the Navier-Stokes volume phase: two blocks of [5][nQ], or the face
// values of six faces
constexpr int kNsG = 10 * knQ > 30 * kn2 ? 10 * knQ : 30 * kn2;

// Kernel families: the phases of a stage, the Navier-Stokes volume phase, and
// the one-shot maps (projection, evaluation, conversions, trace rebuilds).
enum Family { kStage = 0, kNs = 1, kMisc = 2 };

// Resident blocks per SM the registers are limited to.  The stage phases wait
// for latencies (tables, barriers, dependent multiply-adds), so warps count for
// more than a few spilled registers: 16^3 mixed N = 4, two steps, 5.83 / 5.63 /
// 5.52 ms with 6 / 7 / 8 blocks; N = 5 and 6 are limited by shared memory.
constexpr int kStageBlocks = kn <= 5 ? 8 : 5, kNsBlocks = kn <= 5 ? 6 : (kn == 6 ? 4 : 2);
// The split-form volume term holds the states of a line in registers and shared
// memory limits it anyway.  One step of hexahedra, 4 / 5 / 8 blocks: n = 2
// (16^3) 1339 / 1174 / 1163 us, n = 3 (12^3) 1046 / 1040 / 1163 and 928 with 6,
// n = 4 (10^3) 1016 / 1111 / 1252, n = 5 (9^3) 2088 / 1563 / 1569: four are the
// faster there while the last wave is full (10^3 mixed 1396 / 1668 / 1678), five
// never lose to the FP64 kernel (1635 and 2001).
constexpr int kSplitBlocks = kn <= 3 ? 6 : (kn == 4 ? 4 : 5);

// ------------------------------------------------------------------ element phases
//
// The contractions run on the integer pipe (dg_fixed.cuh); what stays on FP64
// is the pointwise physics and the conversions.  Buffers are [var][point] with
// a var stride of nQ.  The few FP64 dot products left carry the 5 variables in
// registers, so one coefficient load feeds 5 independent FMA chains.

#define DG_FMA5(cf, src, stride, acc)            \
  do {                                           \
    const double _c = (cf);                      \
    const double* _s = (src);                    \
    acc[0] = fma(_c, _s[0], acc[0]);             \
    acc[1] = fma(_c, _s[(stride)], acc[1]);      \
    acc[2] = fma(_c, _s[2 * (stride)], acc[2]);  \
    acc[3] = fma(_c, _s[3 * (stride)], acc[3]);  \
    acc[4] = fma(_c, _s[4 * (stride)], acc[4]);  \
  } while (0)

// Modal -> nodal by the sum-factorised passes: sQ [5][nM] (modal
// coefficients) -> U in bufA [5][nQ]; bufB is scratch (sQ may alias it).  IEEE:
// the one-shot maps (fx_wild).
template <bool IEEE>
__device__ __forceinline__ void modal_to_nodal_passes(const Ctx& c, const TypeTab& T, const double* sQ, double* bufA,
                                                      double* bufB) {
  fx_to_nodal<kn, false, IEEE>(c, T, sQ, bufA, bufB, [](int, int, int, double) {});
}

// Storage -> nodal: U = V Q in bufA [5][nQ] from a stored element block sQ.
// A hexahedron is stored as s = W^{1/2} V Q, so U = W^{-1/2} s pointwise;
// the other types hold modal coefficients.  sQ may alias bufB.
template <bool IEEE = false>
__device__ __forceinline__ void modal_to_nodal(const Ctx& c, const TypeTab& T, const double* sQ, double* bufA,
                                            double* bufB, int lane) {
  if (T.type == HEX) {
    constexpr int nQ = knQ;
    const double* rs = c.dpool + T.sqw + nQ;
    for (int w = lane; w < 5 * nQ; w += blockDim.x) bufA[w] = sQ[w] * rs[w % nQ];
    __syncthreads();
    return;
  }
  modal_to_nodal_passes<IEEE>(c, T, sQ, bufA, bufB);
}

// What the nodal->modal pass does with r = M_ref^{-1} V^T bufA of a mode
// (r = V^T bufA without the mass matrix when minv == false):
//   kStore: out[v nM + m] = scale r_v
//   kRk:    K <- a K + scale r (a == 0: K <- scale r; scale includes dt), Q <- Q + b K,
//           and the new Q is also written to sQ when sQ != nullptr.
//   kAxpy:  out[v nM + m] += scale r_v
struct Epilogue {
  enum { kStore = 0, kRk = 1, kAxpy = 2 };
  int kind;
  bool minv;
  double scale;
  double* out;
  const double* Qi;
  double* Qo;
  double* K;
  double* sQ;
  double a, b;
  // curved prism / pyramid: r = Md (V^T bufA) with the element's dense
  // inverse mass matrix Md [nM][nM] (symmetric) instead of minv and scale;
  // rbuf [5][nM] is shared scratch that no other argument aliases
  const double* Md = nullptr;
  double* rbuf = nullptr;
  // true: r is the modal result for a hexahedron too (the conversion to the
  // caller's layout); false: a hexahedron's r is in its scaled nodal storage
  bool modal = false;
};

// The epilogue of one mode given r_v (5 values).  Returns true if a
// non-finite state value was produced.
__device__ __forceinline__ bool epilogue_mode(const Epilogue& ep, int nM, int mode, const double* r) {
  bool bad = false;
  if (ep.kind == Epilogue::kStore) {
#pragma unroll
    for (int v = 0; v < 5; ++v) ep.out[v * nM + mode] = r[v];
  } else if (ep.kind == Epilogue::kAxpy) {
#pragma unroll
    for (int v = 0; v < 5; ++v) ep.out[v * nM + mode] += r[v];
  } else {
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      const int idx = v * nM + mode;
      const double R = r[v];
      const double k = (ep.a == 0.0) ? R : fma(ep.a, ep.K[idx], R);   // r carries dt
      const double qn = fma(ep.b, k, ep.Qi[idx]);
      ep.K[idx] = k;
      ep.Qo[idx] = qn;
      if (ep.sQ) ep.sQ[idx] = qn;
      bad |= !finite_bits(qn);
    }
  }
  return bad;
}

// Applies `ep` to r = V^T h (doubles [5][nM], shared).  Returns true if a
// non-finite state value was produced.
template <bool DENSE>
__device__ __forceinline__ bool finish_modal(const Ctx& c, const TypeTab& T, double* r, int lane,
                                             const Epilogue& ep) {
  const int nM = T.nM;
  const double* dp = c.dpool;
  bool bad = false;
  for (int mode = lane; mode < nM && !DENSE; mode += blockDim.x) {
    double acc[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) acc[v] = r[v * nM + mode];
    const double mi = ep.minv ? dp[T.minv + mode] * ep.scale : ep.scale;
#pragma unroll
    for (int v = 0; v < 5; ++v) acc[v] *= mi;
    bad |= epilogue_mode(ep, nM, mode, acc);
  }
  if (DENSE) {
    dense_product(ep.Md, r, nM, [&](int mode, double* acc) {
#pragma unroll
      for (int v = 0; v < 5; ++v) acc[v] *= ep.scale;
      bad |= epilogue_mode(ep, nM, mode, acc);
    });
  }
  __syncthreads();
  return bad;
}

// Nodal -> modal transpose: bufA [5][nQ] -> modal coefficients through `ep`;
// bufB is scratch.  Returns true if a non-finite state value was produced.
template <bool DENSE, bool IEEE = false>
__device__ __forceinline__ bool nodal_to_modal_t(const Ctx& c, const TypeTab& T, double* bufA, double* bufB, int lane,
                                              const Epilogue& ep) {
  constexpr int nQ = knQ;
  const double* dp = c.dpool;
  const int nM = T.nM;
  if (!DENSE && T.type == HEX && !ep.modal) {
    // scaled nodal storage: W^{1/2} V M^{-1} V^T h = W^{-1/2} h (M = I)
    const double* rs = dp + T.sqw + nQ;
    bool bad = false;
    for (int q = lane; q < nQ; q += blockDim.x) {
      double acc[5];
      const double f = rs[q] * ep.scale;
#pragma unroll
      for (int v = 0; v < 5; ++v) acc[v] = bufA[v * nQ + q] * f;
      bad |= epilogue_mode(ep, nM, q, acc);
    }
    __syncthreads();
    return bad;
  }
  double* r = DENSE ? ep.rbuf : bufB;
  fx_to_modal<kn, IEEE>(T, c, bufA, bufB, r);
  return finish_modal<DENSE>(c, T, r, lane, ep);
}

// ANY: the launch may meet curved elements (their variants are compiled into
// the kernel only then, so affine launches keep the affine register budget).
template <bool ANY, bool IEEE = false>
__device__ __forceinline__ bool nodal_to_modal(const Ctx& c, const TypeTab& T, double* bufA, double* bufB, int lane,
                                               const Epilogue& ep) {
  return (ANY && ep.Md) ? nodal_to_modal_t<true, IEEE>(c, T, bufA, bufB, lane, ep)
                        : nodal_to_modal_t<false, IEEE>(c, T, bufA, bufB, lane, ep);
}

// Values of the nodal field `src` [5][nQ] on the element's own face points
// (neg 0x80000000: negated), written to the face buffer `dst` at the
// element's side slots.
template <int n>
__device__ __forceinline__ void write_traces_n(const TypeTab& T, const int64_t* ft, const double* src, double* dst,
                                            unsigned neg, int ft_mult, int64_t ft_add) {
  fx_traces<n>(T, src, [&](int lf, int v, int p, double x) {
    dst[ft_mult * ft[lf] + ft_add + v * n * n + p] =
        __hiloint2double((int)((unsigned)__double2hiint(x) ^ neg), __double2loint(x));
  });
}

__device__ __forceinline__ void write_traces(const Ctx& c, const TypeTab& T, int64_t s, const double* src,
                                             double* dst, unsigned neg = 0u, int ft_mult = 1, int64_t ft_add = 0) {
  const int64_t* ft = c.slot_ftoff + s * 6;
  write_traces_n<kn>(T, ft, src, dst, neg, ft_mult, ft_add);
}

// Structurally nonzero entries of d(a,b,c)_l / d(xi)_k per type: bit l*3+k.
// hex: diagonal; prism: a(xi, eta); pyramid: a(xi, zeta), b(eta, zeta);
// tet: a(xi, eta, zeta), b(eta, zeta); c = zeta for all.
__constant__ unsigned kMetricMask[4] = {0x111u, 0x113u, 0x135u, 0x137u};

// M = (w_q d(a,b,c)/d(xi)) (J dxi/dx) at volume point q, using each
// collapse's sparsity (hex: diagonal; prism, pyramid, tet: triangular).
__device__ __forceinline__ void point_metric(int type, const double* wa, const double* Jg, double M[3][3]) {
  switch (type) {
    case HEX: {
      double w0 = wa[0];
#pragma unroll
      for (int l = 0; l < 3; ++l)
#pragma unroll
        for (int d = 0; d < 3; ++d) M[l][d] = w0 * Jg[l * 3 + d];
      break;
    }
    case PRISM: {
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        M[0][d] = wa[0] * Jg[d] + wa[1] * Jg[3 + d];
        M[1][d] = wa[4] * Jg[3 + d];
        M[2][d] = wa[8] * Jg[6 + d];
      }
      break;
    }
    case PYR: {
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        M[0][d] = wa[0] * Jg[d] + wa[2] * Jg[6 + d];
        M[1][d] = wa[4] * Jg[3 + d] + wa[5] * Jg[6 + d];
        M[2][d] = wa[8] * Jg[6 + d];
      }
      break;
    }
    default: {  // TET
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        M[0][d] = wa[0] * Jg[d] + wa[1] * Jg[3 + d] + wa[2] * Jg[6 + d];
        M[1][d] = wa[4] * Jg[3 + d] + wa[5] * Jg[6 + d];
        M[2][d] = wa[8] * Jg[6 + d];
      }
      break;
    }
  }
}

// Forward phase of an affine hexahedron in the entropy-stable split form
// (hybridised Gauss SBP operator along every coordinate line):
//   r_i = - sum_j S_ij F#(u_i, u_j) - sum_f s_f E_f,i F#(u_i, u~_f)
//         + sum_f s_f E_f,i sum_j E_f,j F#(u~_f, u_j),
// S = W D - (W D)^T, E_f the extrapolation to the line's end f (s_- = -1,
// s_+ = +1), F# contracted with the line direction's metric J dxi_l/dx, u~_f
// the entropy-projected face state u(E_f v(u)); H_q = sum_l w_perp r_q^(l)
// with w_perp the product of the two other directions' weights.  For a
// central F# this is the weak form's H (sum_l D_l^T G_l).  The face states
// u~ are this element's traces (the face kernel takes the Riemann flux on
// them).  Every unordered node pair and every (face state, node) pair of a
// line is evaluated once per direction (F# is symmetric) into shared memory,
// then every node sums its line's terms.  sQ lives at the start of bufG;
// workspace: bufA [5 nQ] (nodal state, then entropy variables, then the
// accumulated H), bufG: [kTP][nQ] two-point quantities, [kTP][6 n^2] of the
// face states, then one direction's [n^2][n(n-1)/2][5] pair fluxes and
// [n^2][2][n][5] face-state fluxes.
__device__ __forceinline__ void element_forward_split(const Ctx& c, const TypeTab& T, int64_t s, double* bufA,
                                                   double* bufG, int lane) {
  constexpr int n = kn, nQ = knQ, n2 = kn2, nF = 6 * n2;
  const double* dp = c.dpool;
  const double gamma = c.gamma, gm1 = gamma - 1.0, igm1 = 1.0 / gm1;
  modal_to_nodal(c, T, bufG, bufA, bufG, lane);
  double* P = bufG;
  double* Pf = P + kTP * nQ;
  double* Gs = Pf + kTP * nF;
  // nodal two-point quantities; the entropy variables overwrite U in place
  for (int q = lane; q < nQ; q += blockDim.x) {
    double U[5], Pq[kTP], v[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) U[k] = bufA[k * nQ + q];
    two_point_state(U, gm1, Pq);
#pragma unroll
    for (int k = 0; k < kTP; ++k) P[k * nQ + q] = Pq[k];
    entropy_variables(Pq, 1, gamma, v);
#pragma unroll
    for (int k = 0; k < 5; ++k) bufA[k * nQ + q] = v[k];
  }
  __syncthreads();
  // entropy-projected face states: extrapolate v along the face-normal
  // coordinate, map back; they are the element's traces
  const int64_t* ft = c.slot_ftoff + s * 6;
  for (int w = lane; w < nF; w += blockDim.x) {
    const int lf = w / n2, p = w - lf * n2;
    const int ia = p % n, ib = p / n;
    const FaceDesc d = T.faces[lf];
    const int sa = d.alpha == 0 ? n2 : (d.alpha == 1 ? n : 1);
    const int sb = d.beta == 0 ? n2 : (d.beta == 1 ? n : 1);
    const int sf = d.fixed == 0 ? n2 : (d.fixed == 1 ? n : 1);
    const double* e = dp + T.ext + d.end * n;
    const double* V = bufA + ia * sa + ib * sb;
    double vt[5] = {0, 0, 0, 0, 0};
    for (int m = 0; m < n; ++m) DG_FMA5(e[m], V + m * sf, nQ, vt);
    double U[5], Pp[kTP];
    from_entropy_variables(vt, gamma, U, Pp);
    double* out = c.T + ft[lf] + p;
#pragma unroll
    for (int k = 0; k < 5; ++k) out[k * n2] = U[k];
#pragma unroll
    for (int k = 0; k < kTP; ++k) Pf[k * nF + w] = Pp[k];
  }
  __syncthreads();
  const ElemGeo& g = c.geo[s];
  const double* S = dp + T.sbp;
  const double* w1 = dp + T.w1;
  const double* E = dp + T.ext;
  const int np = n * (n - 1) / 2;         // unordered node pairs of a line
  double* Fp = Gs;                        // [n^2 lines][np][5] pair fluxes of one direction
  double* Ff = Fp + (size_t)n2 * np * 5;  // [n^2 lines][2 ends][n][5] face-state fluxes of one direction
  // the local face at the end `end` of coordinate l, and the index of a face
  // point from the two other coordinates' indices (x1 < x2 by coordinate)
  auto face_of = [&](int l, int end) {
    int lf = 0;
    for (int k = 0; k < 6; ++k)
      if (T.faces[k].fixed == l && T.faces[k].end == end) lf = k;
    return lf;
  };
  auto face_point = [&](int lf, int l, int x1, int x2) {
    const FaceDesc d = T.faces[lf];
    const int o1 = l == 0 ? 1 : 0;
    const int ia = d.alpha == o1 ? x1 : x2, ib = d.beta == o1 ? x1 : x2;
    return lf * n2 + ia + ib * n;
  };
  // H accumulates in bufA (the entropy variables are no longer needed)
  for (int w = lane; w < 5 * nQ; w += blockDim.x) bufA[w] = 0.0;
  const int st[3] = {n2, n, 1};
#pragma unroll 1
  for (int l = 0; l < 3; ++l) {
    const int o1 = l == 0 ? 1 : 0, o2 = l == 2 ? 1 : 2;
    const double m[3] = {g.Jg[3 * l], g.Jg[3 * l + 1], g.Jg[3 * l + 2]};
    const int lf_end[2] = {face_of(l, 0), face_of(l, 1)};
    // every unordered node pair and every (face state, node) pair of every
    // line of this direction once (F# is symmetric)
    const int tasks = n2 * (np + 2 * n);
    for (int t = lane; t < tasks; t += blockDim.x) {
      double F[5];
      int line, k;
      if (t < n2 * np) {
        line = t / np;
        k = t - line * np;
        int i = 0, kk = k;
        while (kk >= n - 1 - i) {
          kk -= n - 1 - i;
          ++i;
        }
        const int j = i + 1 + kk;
        const int x1 = line / n, x2 = line - x1 * n;
        const int base = x1 * st[o1] + x2 * st[o2];
        two_point_flux(P + base + i * st[l], nQ, P + base + j * st[l], nQ, m, igm1, F);
        double* out = Fp + ((size_t)line * np + k) * 5;
#pragma unroll
        for (int v = 0; v < 5; ++v) out[v] = F[v];
      } else {
        const int u = t - n2 * np;
        line = u / (2 * n);
        const int rem = u - line * 2 * n, end = rem / n, j = rem - end * n;
        const int x1 = line / n, x2 = line - x1 * n;
        const int base = x1 * st[o1] + x2 * st[o2];
        two_point_flux(Pf + face_point(lf_end[end], l, x1, x2), nF, P + base + j * st[l], nQ, m, igm1, F);
        double* out = Ff + (((size_t)line * 2 + end) * n + j) * 5;
#pragma unroll
        for (int v = 0; v < 5; ++v) out[v] = F[v];
      }
    }
    __syncthreads();
    // per node: the line's terms of this direction
    for (int q = lane; q < nQ; q += blockDim.x) {
      const int idx[3] = {q / n2, (q / n) % n, q % n};
      const int x1 = idx[o1], x2 = idx[o2], ii = idx[l];
      const int line = x1 * n + x2;
      const double* Fl = Fp + (size_t)line * np * 5;
      double r[5] = {0, 0, 0, 0, 0};
      for (int j = 0; j < n; ++j) {
        if (j == ii) continue;
        const int i0 = ii < j ? ii : j, j0 = ii < j ? j : ii;
        const double* F = Fl + (i0 * (2 * n - i0 - 1) / 2 + (j0 - i0 - 1)) * 5;
        const double sij = -S[ii * n + j];
#pragma unroll
        for (int k = 0; k < 5; ++k) r[k] = fma(sij, F[k], r[k]);
      }
#pragma unroll
      for (int end = 0; end < 2; ++end) {
        const double* Fe = Ff + ((size_t)line * 2 + end) * n * 5;
        double G[5] = {0, 0, 0, 0, 0};
        for (int j = 0; j < n; ++j) {
          const double ej = E[end * n + j];
#pragma unroll
          for (int k = 0; k < 5; ++k) G[k] = fma(ej, Fe[j * 5 + k], G[k]);
        }
        const double se = (end ? 1.0 : -1.0) * E[end * n + ii];
#pragma unroll
        for (int k = 0; k < 5; ++k) r[k] = fma(se, G[k] - Fe[ii * 5 + k], r[k]);
      }
      const double wp = w1[x1] * w1[x2];
#pragma unroll
      for (int k = 0; k < 5; ++k) bufA[k * nQ + q] = fma(wp, r[k], bufA[k * nQ + q]);
    }
    __syncthreads();
  }
  double* H = c.H + c.slot_hoff[s];
  for (int w = lane; w < 5 * nQ; w += blockDim.x) H[w] = bufA[w];
  __syncthreads();
}

// Forward phase of the element at slot s: nodal state, own-face traces and
// the nodal volume residual H.  sQ lives at the start of bufG.
template <bool ANY>
__device__ __forceinline__ void element_forward_t(const Ctx& c, const TypeTab& T, int64_t s, double* bufA, double* bufG,
                                                  int lane) {
  constexpr int nQ = knQ;
  const double* dp = c.dpool;
  if (T.type == HEX) {
    modal_to_nodal(c, T, bufG, bufA, bufG, lane);
    write_traces(c, T, s, bufA, c.T);
  } else {
    const int64_t* ft = c.slot_ftoff + s * 6;
    fx_to_nodal<kn, true, false>(c, T, bufG, bufA, bufG,
                          [&](int lf, int v, int p, double x) { c.T[__ldg(ft + lf) + v * kn2 + p] = x; });
  }
  if (c.Usave) {
    // kept for the adjoint (reverse LSERK with stored stage data)
    double* Un = c.Usave + c.slot_hoff[s];
    for (int w = lane; w < 5 * nQ; w += blockDim.x) Un[w] = bufA[w];
  }
  if (c.ns) {
    // Navier-Stokes: the volume residual needs the lifted gradient, which
    // needs the neighbours' traces; keep the nodal state for that phase.
    double* Un = c.Unod + c.slot_hoff[s];
    for (int w = lane; w < 5 * nQ; w += blockDim.x) Un[w] = bufA[w];
    __syncthreads();
    return;
  }
  // contravariant fluxes G_l at the volume points (bufG, [3][5][nQ])
  const ElemGeo& g = c.geo[s];
  double Jg[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) Jg[k] = g.Jg[k];
  // a curved element reads its pointwise metric w (da/dxi)(J dxi/dx) instead
  const bool curved = ANY && c.slot_coff[s] >= 0;
  const double* cm = curved ? c.cpool + c.slot_coff[s] : nullptr;
  // moving mesh: the mesh velocity at the volume points
  const double* xd = (curved && c.mpool) ? c.mpool + c.slot_moff[s] + 31 * nQ : nullptr;
  const double gm1 = c.gamma - 1.0;
  auto put = [&](double* G, int v, double x) { G[v * nQ] = x; };
  for (int q = lane; q < nQ; q += blockDim.x) {
    double U[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) U[v] = bufA[v * nQ + q];
    double M[3][3];
    if (ANY && curved) {
#pragma unroll
      for (int l = 0; l < 3; ++l)
#pragma unroll
        for (int d = 0; d < 3; ++d) M[l][d] = cm[(l * 3 + d) * nQ + q];
    } else {
      point_metric(T.type, dp + T.wA + q * 9, Jg, M);
    }
    double rinv = rcp(U[0]);
    double u = U[1] * rinv, v = U[2] * rinv, w = U[3] * rinv;
    double p = gm1 * (U[4] - 0.5 * (U[1] * u + U[2] * v + U[3] * w));
    double Ep = U[4] + p;
    if (ANY && xd) {
      // moving frame: (F(U) - U xdot) through the metric, W_l = M_l . xdot
      const double x0 = xd[q], x1 = xd[nQ + q], x2 = xd[2 * nQ + q];
#pragma unroll
      for (int l = 0; l < 3; ++l) {
        const double Vl = M[l][0] * u + M[l][1] * v + M[l][2] * w;
        const double Rl = Vl - (M[l][0] * x0 + M[l][1] * x1 + M[l][2] * x2);
        double* G = bufG + l * 5 * nQ + q;
        put(G, 0, Rl * U[0]);
        put(G, 1, Rl * U[1] + p * M[l][0]);
        put(G, 2, Rl * U[2] + p * M[l][1]);
        put(G, 3, Rl * U[3] + p * M[l][2]);
        put(G, 4, Rl * U[4] + Vl * p);
      }
      continue;
    }
#pragma unroll
    for (int l = 0; l < 3; ++l) {
      double Vl = M[l][0] * u + M[l][1] * v + M[l][2] * w;
      double* G = bufG + l * 5 * nQ + q;
      put(G, 0, Vl * U[0]);
      put(G, 1, Vl * U[1] + p * M[l][0]);
      put(G, 2, Vl * U[2] + p * M[l][1]);
      put(G, 3, Vl * U[3] + p * M[l][2]);
      put(G, 4, Vl * Ep);
    }
  }
  // H = sum_l D_l^T G_l (collocation derivative along each collapsed direction)
  // (the last direction's sums run in place of its own G)
  __syncthreads();
  fx_dsum<kn>([&](int l, int v, int q) { return bufG[(5 * l + v) * nQ + q]; }, 7u, bufG + 10 * nQ,
              c.H + c.slot_hoff[s]);
}

template <bool ANY, bool SPLIT>
__device__ __forceinline__ void element_forward(const Ctx& c, const TypeTab& T, int64_t s, double* bufA, double* bufG,
                                                int lane) {
  if (SPLIT && T.type == HEX) element_forward_split(c, T, s, bufA, bufG, lane);
  else element_forward_t<ANY>(c, T, s, bufA, bufG, lane);
}

// Backward phase, first half: bufA = H +- sum_faces E_f^T F_f with the
// face values F_f read from `faces` (the lifted fluxes, subtracted with neg
// 0x80000000; the adjoint's trace cotangents, added with neg 0).  H and F are
// staged into bufG with coalesced loads first (H is read in place for n = 2,
// where bufG holds the face values only).
template <bool ANY>
__device__ __forceinline__ void element_lift(const Ctx& c, const TypeTab& T, int64_t s, double* bufA, double* bufG,
                                            int lane, const double* faces, unsigned neg, const double* pscale) {
  constexpr int nQ = knQ, n2 = kn2;
  constexpr bool room = 30 * n2 + 5 * nQ <= 15 * nQ;
  const int nf = T.nfaces;
  const int64_t* ft = c.slot_ftoff + s * 6;
  const double* H = c.H + c.slot_hoff[s];
  double* sH = bufG + 30 * n2;
  for (int w = lane; w < 5 * nQ && room; w += blockDim.x) sH[w] = H[w];
#pragma unroll
  for (int v = 0; v < 5; ++v)
    for (int w = lane; w < nf * n2; w += blockDim.x) {
      const int lf = w / n2, o = v * n2 + w - lf * n2;
      bufG[lf * 5 * n2 + o] = faces[ft[lf] + o];
    }
  __syncthreads();
  fx_lift<kn>(T, [&](int o) { return room ? sH[o] : H[o]; }, bufG, neg, bufA, [&](int o, double x) {
    // curved hexahedron: M^{-1} V^T = V^T diag(1/J) (V square, V^T W V = I)
    bufA[o] = ANY && pscale ? x * pscale[o % nQ] : x;
  });
}

// Backward phase of the element: r = V^T (H +- sum_f E_f^T F_f) through `ep`.
// pscale: a curved hexahedron's pointwise 1/J before V^T, or null.  Returns
// true if a non-finite state value was produced.
template <bool ANY>
__device__ __forceinline__ bool element_backward(const Ctx& c, const TypeTab& T, int64_t s, double* bufA, double* bufG,
                                                 int lane, const double* faces, unsigned neg, const double* pscale,
                                                 const Epilogue& ep) {
  if (T.type == HEX) {
    element_lift<ANY>(c, T, s, bufA, bufG, lane, faces, neg, pscale);
    return nodal_to_modal_t<false>(c, T, bufA, bufG, lane, ep);
  }
  double* r = ANY && ep.Md ? ep.rbuf : bufA;
  const double* H = c.H + c.slot_hoff[s];
  const int64_t* ft = c.slot_ftoff + s * 6;
  fx_lift_to_modal<kn, true>(c, T, [&](int o) { return H[o]; },
                       [&](int lf, int v, int p) { return faces[__ldg(ft + lf) + v * kn2 + p]; }, neg, bufA, bufG, r);
  return ANY && ep.Md ? finish_modal<true>(c, T, r, lane, ep) : finish_modal<false>(c, T, r, lane, ep);
}

// BR1 lifting face term of a hexahedron: out(o, dW(o) - sum_f n_d(f) E_f^T L_f),
// n(f) the element's outward unit normal of local face f and L_f the face
// values at its own points (staged through bufS; bufA scratch).
template <bool CURVED, class Out>
__device__ __forceinline__ void lift_scaled_t(const Ctx& c, const TypeTab& T, int64_t s, const double* dW, double* bufA,
                                           double* bufS, int lane, const double* faces, int d, Out out) {
  constexpr int n2 = kn2;
  const int nf = T.nfaces;
  const int64_t* ft = c.slot_ftoff + s * 6;
  // the normal multiplies the staged face values (curved: point by point,
  // c.snrm holds each side's own normals)
#pragma unroll
  for (int v = 0; v < 5; ++v)
    for (int w = lane; w < nf * n2; w += blockDim.x) {
      const int lf = w / n2, p = w - lf * n2, o = v * n2 + p;
      const double nd = CURVED ? c.snrm[3 * (ft[lf] / 5) + d * n2 + p] : c.fnrm[(s * 6 + lf) * 3 + d];
      bufS[lf * 5 * n2 + o] = nd * faces[ft[lf] + o];
    }
  __syncthreads();
  fx_lift<kn>(T, [&](int o) { return dW[o]; }, bufS, 0x80000000u, bufA, out);
}

// Navier-Stokes volume phase of the element at slot s (after the lifting face
// phase).  Per direction d the BR1 lifted gradient of W = (rho, u, v, w, p):
//   nodal  Hd = sum_l D_l^T (w J da_l/dx_d W)          (volume term, as H)
//   modal  G_d = -(1/J) M_ref^{-1} V^T (Hd - sum_f n_d(f) E_f^T L_f)
//   nodal  grad_d W = V G_d, and its traces on the own face points (Vt);
// then the total flux F_e(U) - F_v(U, grad W) at the volume points and
// H = sum_l D_l^T G_l(F) as in the Euler forward phase.
// smem: bufA [5 nQ] | bufDW [3][5][nQ] | bufG [kNsG].  The products with the
// metric are formed where a derivative pass reads them and the total flux
// overwrites the gradient, so an element takes 30 nQ doubles (40 with buffers of
// their own: fewer resident blocks, and the phase waits for latencies).
template <bool CURVED>
__device__ __forceinline__ void element_ns_volume_t(const Ctx& c, const TypeTab& T, int64_t s, double* smem, int lane) {
  constexpr int nQ = knQ, n2 = kn2;
  // curved element: pointwise metric [9][nQ], J, 1/J, (prism, pyramid) dense M_e^{-1}
  const double* cblk = CURVED ? c.cpool + c.slot_coff[s] : nullptr;
  constexpr int nQm = knQ;
  double* bufA = smem;
  double* bufDW = smem + 5 * nQm;
  double* bufG = smem + 20 * nQm;
  const double* Un = c.Unod + c.slot_hoff[s];
  const double* dp = c.dpool;
  const double gm1 = c.gamma - 1.0;
  const ElemGeo& g = c.geo[s];
  double Jg[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) Jg[k] = g.Jg[k];
  // moving mesh (lift_phase != 0): prisms and pyramids split at the lifting's
  // M(t)^{-1}; hexahedra run whole in phase 2
  const bool dense_split = CURVED && c.lift_phase != 0 && T.type != HEX;
  if (CURVED && c.lift_phase == 1 && !dense_split) return;
  if (dense_split && c.lift_phase == 2) {
    // the solved modal gradient of every direction: nodal values, traces
    for (int d = 0; d < 3; ++d) {
      double* dW = bufDW + d * 5 * nQ;
      const double* Gm = c.lift + (int64_t)d * c.lift_stride + c.slot_qoff[s];
      double* sG = bufG + 5 * nQ;
      for (int w = lane; w < 5 * T.nM; w += blockDim.x) sG[w] = Gm[w];
      __syncthreads();
      const int64_t* ft = c.slot_ftoff + s * 6;
      fx_to_nodal<kn, true, false>(c, T, sG, dW, bufG, [&](int lf, int v, int p, double x) {
        c.Vt[3 * __ldg(ft + lf) + (d * 5 + v) * n2 + p] = x;
      });
    }
  } else {
  // Lifting volume terms through the reference directions: with
  // M[l][d] = sum_k wA[l][k] Jg[k][d] (wA = w da_l/dxi_k, structurally sparse
  // per type), Hd = sum_l D_l^T (M[l][d] W) = sum_k Jg[k][d] P_k with
  // P_k = sum_{l: wA[l][k] != 0} D_l^T (wA[l][k] W): 3 (hex) to 6 (tet)
  // directional passes instead of 9.  H_0..H_2 accumulate in bufDW.
  for (int q = lane; q < nQ; q += blockDim.x) {
    double U[5], W[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) U[v] = Un[v * nQ + q];
    primitive(U, gm1, W);
#pragma unroll
    for (int v = 0; v < 5; ++v) bufA[v * nQ + q] = W[v];
  }
  const unsigned nz = kMetricMask[T.type];
#pragma unroll 1
  for (int k = 0; k < 3; ++k) {
    // affine: P_k; a curved element takes one full set of directional passes
    // per direction with its pointwise metric, H_d = sum_l D_l^T (M_q[l][d] W)
    const unsigned dirs = CURVED ? 7u : ((nz >> k) & 1u) | (((nz >> (3 + k)) & 1u) << 1) | (((nz >> (6 + k)) & 1u) << 2);
    auto metric = [&](int l, int q) {
      return CURVED ? cblk[(l * 3 + k) * nQ + q] : __ldg(dp + T.wA + q * 9 + l * 3 + k);
    };
    __syncthreads();
    fx_dsum<kn>([&](int l, int v, int q) { return metric(l, q) * bufA[v * nQ + q]; }, dirs, bufG + 5 * nQ,
                CURVED ? bufDW + k * 5 * nQ : bufG);
    if (!CURVED) {
      for (int w = lane; w < 5 * nQ; w += blockDim.x) {
        const double p = bufG[w];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          double* Hd = bufDW + d * 5 * nQ + w;
          const double jkd = Jg[k * 3 + d];
          *Hd = k == 0 ? jkd * p : fma(jkd, p, *Hd);
        }
      }
      __syncthreads();
    }
  }
#pragma unroll 1
  for (int d = 0; d < 3; ++d) {
    double* dW = bufDW + d * 5 * nQ;
    if (T.type == HEX) {
      // V is square for the hexahedron, so V M^{-1} V^T = (W J)^{-1}: the
      // projection onto the modal space is the identity at the nodes
      const double* wq = dp + T.W;
      const double* iJ = CURVED ? cblk + 10 * nQ : nullptr;
      lift_scaled_t<CURVED>(c, T, s, dW, bufA, bufG, lane, c.L, d, [&](int o, double x) {
        dW[o] = -(CURVED ? iJ[o % nQ] : g.invJ) * x * rcp(wq[o % nQ]);
      });
      write_traces(c, T, s, dW, c.Vt, 0u, 3, (int64_t)d * 5 * n2);
    } else {
      // r = V^T (Hd - sum_f n_d(f) E_f^T L_f), then the projection
      const int64_t* ft = c.slot_ftoff + s * 6;
      fx_lift_to_modal<kn, false>(
          c, T, [&](int o) { return dW[o]; },
          [&](int lf, int v, int p) {
            const int64_t t = __ldg(ft + lf);
            const double nd = CURVED ? c.snrm[3 * (t / 5) + d * n2 + p] : c.fnrm[(s * 6 + lf) * 3 + d];
            return nd * c.L[t + v * n2 + p];
          },
          0x80000000u, bufA, bufG, bufA);
      if (dense_split) {
        // phase 1: r_d = -V^T (lifting terms); M(t)^{-1} r_d is solved outside
        Epilogue ep{Epilogue::kStore, false, -1.0, c.lift + (int64_t)d * c.lift_stride + c.slot_qoff[s], nullptr,
                    nullptr, nullptr, nullptr, 0.0, 0.0};
        finish_modal<false>(c, T, bufA, lane, ep);
        continue;
      }
      double* sG = bufG + 5 * nQ;
      Epilogue ep{Epilogue::kStore, true, CURVED ? -1.0 : -g.invJ, sG, nullptr, nullptr, nullptr, nullptr, 0.0, 0.0};
      if (CURVED) ep.Md = cblk + 11 * nQ;
      finish_modal<CURVED>(c, T, bufA, lane, ep);
      fx_to_nodal<kn, true, false>(c, T, sG, dW, bufG, [&](int lf, int v, int p, double x) {
        c.Vt[3 * __ldg(ft + lf) + (d * 5 + v) * n2 + p] = x;
      });
    }
    if (c.DW) {
      double* out = c.DW + 3 * c.slot_hoff[s] + d * 5 * nQ;
      for (int w = lane; w < 5 * nQ; w += blockDim.x) out[w] = dW[w];
    }
    __syncthreads();
  }
  if (dense_split) return;   // phase 1 ends with the lifting residuals
  }
  // total contravariant flux G_l = sum_d M[l][d] (F_e - F_v)_d
  // (in place of the point's gradient)
  __syncthreads();
  auto put = [&](double* G, int v, double x) { G[v * nQ] = x; };
  for (int q = lane; q < nQ; q += blockDim.x) {
    double U[5], W[5], gr[15];
#pragma unroll
    for (int v = 0; v < 5; ++v) U[v] = Un[v * nQ + q];
#pragma unroll
    for (int t = 0; t < 15; ++t) gr[t] = bufDW[t * nQ + q];
    primitive(U, gm1, W);
    double Fv[3][5];
    viscous_flux(W, gr, c.mu, c.kappa, Fv);
    double M[3][3];
    if (CURVED) {
#pragma unroll
      for (int l = 0; l < 3; ++l)
#pragma unroll
        for (int dd = 0; dd < 3; ++dd) M[l][dd] = cblk[(l * 3 + dd) * nQ + q];
    } else {
      point_metric(T.type, dp + T.wA + q * 9, Jg, M);
    }
    const double u = W[1], v = W[2], w = W[3], p = W[4], Ep = U[4] + p;
    if (CURVED && c.mpool) {
      // moving mesh: the convective flux in the moving frame, F(U) - U xdot
      const double* xd = c.mpool + c.slot_moff[s] + 31 * nQ;
      const double x0 = xd[q], x1 = xd[nQ + q], x2 = xd[2 * nQ + q];
#pragma unroll
      for (int l = 0; l < 3; ++l) {
        const double Vl = M[l][0] * u + M[l][1] * v + M[l][2] * w;
        const double Rl = Vl - (M[l][0] * x0 + M[l][1] * x1 + M[l][2] * x2);
        double* G = bufDW + l * 5 * nQ + q;
        put(G, 0, Rl * U[0]);
        put(G, 1, Rl * U[1] + p * M[l][0] - (M[l][0] * Fv[0][1] + M[l][1] * Fv[1][1] + M[l][2] * Fv[2][1]));
        put(G, 2, Rl * U[2] + p * M[l][1] - (M[l][0] * Fv[0][2] + M[l][1] * Fv[1][2] + M[l][2] * Fv[2][2]));
        put(G, 3, Rl * U[3] + p * M[l][2] - (M[l][0] * Fv[0][3] + M[l][1] * Fv[1][3] + M[l][2] * Fv[2][3]));
        put(G, 4, Rl * U[4] + Vl * p - (M[l][0] * Fv[0][4] + M[l][1] * Fv[1][4] + M[l][2] * Fv[2][4]));
      }
      continue;
    }
#pragma unroll
    for (int l = 0; l < 3; ++l) {
      double Vl = M[l][0] * u + M[l][1] * v + M[l][2] * w;
      double* G = bufDW + l * 5 * nQ + q;
      put(G, 0, Vl * U[0]);
      put(G, 1, Vl * U[1] + p * M[l][0] - (M[l][0] * Fv[0][1] + M[l][1] * Fv[1][1] + M[l][2] * Fv[2][1]));
      put(G, 2, Vl * U[2] + p * M[l][1] - (M[l][0] * Fv[0][2] + M[l][1] * Fv[1][2] + M[l][2] * Fv[2][2]));
      put(G, 3, Vl * U[3] + p * M[l][2] - (M[l][0] * Fv[0][3] + M[l][1] * Fv[1][3] + M[l][2] * Fv[2][3]));
      put(G, 4, Vl * Ep - (M[l][0] * Fv[0][4] + M[l][1] * Fv[1][4] + M[l][2] * Fv[2][4]));
    }
  }
  __syncthreads();
  fx_dsum<kn>([&](int l, int v, int q) { return bufDW[(5 * l + v) * nQ + q]; }, 7u, bufG, c.H + c.slot_hoff[s]);
}

template <bool ANY>
__device__ __forceinline__ void element_ns_volume(const Ctx& c, const TypeTab& T, int64_t s, double* smem, int lane) {
  if (ANY && c.slot_coff[s] >= 0) element_ns_volume_t<true>(c, T, s, smem, lane);
  else element_ns_volume_t<false>(c, T, s, smem, lane);
}

// One element at slot s.  smem per block: bufA [5 nQ], bufG [15 nQ]
// (30 nQ for the Navier-Stokes volume phase).
template <int FAM, bool ANY, bool SPLIT>
__device__ __forceinline__ void process_element(const Ctx& c, int mode, const StageArgs& io, int64_t s, double* bufA,
                                                double* bufG, int lane) {
  const TypeTab& T = c.tabs[c.slot_tab[s]];
  constexpr int nQ = knQ;
  const int nM = T.nM;
  const int64_t qoff = c.slot_qoff[s];
  if constexpr (FAM == kNs) {
    element_ns_volume<ANY>(c, T, s, bufA, lane);
    return;
  }
  if constexpr (FAM == kMisc) if (mode == kGather) {
    // hexahedra only: caller modal coefficients Q -> storage s = W^{1/2} V Q
    const double* Q = io.Qin + c.elem_qoff[c.elem_of_slot[s]];
    for (int w = lane; w < 5 * nM; w += blockDim.x) bufG[w] = Q[w];
    __syncthreads();
    modal_to_nodal_passes<true>(c, T, bufG, bufA, bufG);
    const double* sq = c.dpool + T.sqw;
    double* out = io.Qout + qoff;
    for (int w = lane; w < 5 * nQ; w += blockDim.x) out[w] = bufA[w] * sq[w % nQ];
    __syncthreads();
    return;
  }
  if constexpr (FAM == kMisc) if (mode == kScatter) {
    // hexahedra only: storage s -> caller modal coefficients V^{-1} W^{-1/2} s = V^T (w W^{-1/2}) s
    const double* S = io.Qin + qoff;
    const double* sq = c.dpool + T.sqw + 2 * nQ;
    for (int w = lane; w < 5 * nQ; w += blockDim.x) bufA[w] = S[w] * sq[w % nQ];
    __syncthreads();
    Epilogue ep{Epilogue::kStore, false, 1.0, io.Qout + c.elem_qoff[c.elem_of_slot[s]], nullptr, nullptr, nullptr,
                nullptr, 0.0, 0.0};
    ep.modal = true;
    nodal_to_modal_t<false, true>(c, T, bufA, bufG, lane, ep);
    return;
  }
  if constexpr (FAM == kStage) if (mode == kFwd) {
    const double* Q = io.Qin + qoff;
    for (int w = lane; w < 5 * nM; w += blockDim.x) bufG[w] = Q[w];
    __syncthreads();
    element_forward<ANY, SPLIT>(c, T, s, bufA, bufG, lane);
    return;
  }
  if constexpr (FAM == kMisc) if (mode == kTraces) {
    // the stage's face traces rebuilt from its kept nodal state (and the
    // gradient traces from its kept nodal gradient) by the same trace
    // writes as the forward phases: bitwise the values they wrote
    const double* Un = c.Unod + c.slot_hoff[s];
    for (int w = lane; w < 5 * nQ; w += blockDim.x) bufA[w] = Un[w];
    __syncthreads();
    write_traces(c, T, s, bufA, c.T);
    if (c.ns) {
      for (int d = 0; d < 3; ++d) {
        const double* dW = c.DW + 3 * c.slot_hoff[s] + d * 5 * nQ;
        __syncthreads();
        for (int w = lane; w < 5 * nQ; w += blockDim.x) bufG[w] = dW[w];
        __syncthreads();
        write_traces(c, T, s, bufG, c.Vt, 0u, 3, (int64_t)d * 5 * kn2);
      }
    }
    __syncthreads();
    return;
  }
  if constexpr (FAM == kMisc) if (mode == kEval) {
    const double* Q = io.Qin + qoff;
    for (int w = lane; w < 5 * nM; w += blockDim.x) bufG[w] = Q[w];
    __syncthreads();
    modal_to_nodal<true>(c, T, bufG, bufA, bufG, lane);
    double* out = io.Qout + c.elem_voff[c.elem_of_slot[s]];
    for (int w = lane; w < 5 * nQ; w += blockDim.x) out[w] = bufA[w];
    __syncthreads();
    return;
  }
  // Curved element: pointwise J (cpool block [9][nQ] metric, [nQ] J, [nQ] 1/J,
  // then for prism / pyramid the dense M_e^{-1}); the affine scale 1/J_e and
  // the diagonal M_ref^{-1} are replaced by diag(1/J_q) before V^T (hex) or by
  // M_e^{-1} after it (prism, pyramid).  Tetrahedra are always affine.
  const int64_t coff = ANY && c.slot_coff ? c.slot_coff[s] : -1;
  const double* cblk = coff >= 0 ? c.cpool + coff : nullptr;
  // moving mesh: the backward phase returns vol - surf itself (the rate of
  // the mass-weighted state; the mass matrix is solved separately)
  const bool moving = ANY && c.mpool != nullptr;
  const bool dense = cblk && T.type != HEX && (!moving || FAM == kMisc);
  if constexpr (FAM == kMisc) if (mode == kLoad) {
    // b = V^T W J q: pointwise J_q (curved) or the element's constant J
    const int64_t e = c.elem_of_slot[s];
    const double* vals = io.Qin + c.elem_voff[e];
    const double* W = c.dpool + T.W;
    if (cblk) {
      const double* Jq = cblk + 9 * nQ;
      for (int w = lane; w < 5 * nQ; w += blockDim.x) bufA[w] = W[w % nQ] * Jq[w % nQ] * vals[w];
    } else {
      for (int w = lane; w < 5 * nQ; w += blockDim.x) bufA[w] = W[w % nQ] * vals[w];
    }
    __syncthreads();
    Epilogue ep{Epilogue::kStore, false, cblk ? 1.0 : 1.0 / c.geo[s].invJ, io.Qout + qoff, nullptr, nullptr, nullptr,
                nullptr, 0.0, 0.0};
    nodal_to_modal<false, true>(c, T, bufA, bufG, lane, ep);
    return;
  }
  if constexpr (FAM == kMisc) if (mode == kProject) {
    const int64_t e = c.elem_of_slot[s];
    const double* vals = io.Qin + c.elem_voff[e];
    const double* W = c.dpool + T.W;
    if (dense) {
      const double* Jq = cblk + 9 * nQ;
      for (int w = lane; w < 5 * nQ; w += blockDim.x) bufA[w] = W[w % nQ] * Jq[w % nQ] * vals[w];
    } else {
      for (int w = lane; w < 5 * nQ; w += blockDim.x) bufA[w] = W[w % nQ] * vals[w];
    }
    __syncthreads();
    Epilogue ep{Epilogue::kStore, true, 1.0, io.Qout + qoff, nullptr, nullptr, nullptr, nullptr, 0.0, 0.0};
    if (dense) {
      ep.Md = cblk + 11 * nQ;
      ep.rbuf = bufG + 5 * nQ;
    }
    nodal_to_modal<ANY, true>(c, T, bufA, bufG, lane, ep);
    return;
  }
  if constexpr (FAM == kStage) {
    const double* pscale = (cblk && T.type == HEX && !moving) ? cblk + 10 * nQ : nullptr;
    const double invJ = cblk ? 1.0 : c.geo[s].invJ;
    // one epilogue for both kinds of step, so that the backward code exists once
    const bool rhs = mode == kBwdRhs;
    Epilogue ep{rhs ? Epilogue::kStore : Epilogue::kRk, !moving, rhs ? invJ : invJ * io.dt, rhs ? io.Qout + qoff : nullptr, io.Qin + qoff,
                io.Qout + qoff, io.K + qoff, mode == kBwdRkFwd ? bufG : nullptr, io.a, io.b};
    if (dense) {
      ep.Md = cblk + 11 * nQ;
      ep.rbuf = bufG + 5 * nQ;
    }
    const bool bad = __syncthreads_or(element_backward<ANY>(c, T, s, bufA, bufG, lane, c.T, 0x80000000u, pscale, ep));
    if (bad && lane == 0) atomicOr(c.status, 1u);
    if (mode == kBwdRkFwd) element_forward<ANY, SPLIT>(c, T, s, bufA, bufG, lane);
  }
}

// ------------------------------------------------------------------ adjoint element phases
//
// With r = V^T (H - sum_f E_f^T Fhat_f), R = diag(M_ref^-1 / J) r and
// H = sum_l D_l^T G_l(U), U = V Q, the cotangent Rbar maps back as
//   Ybar = V diag(M_ref^-1 / J) Rbar          (nodal, a modal->nodal pass)
//   seed_f = -E_f Ybar                         (cotangent of Fhat_f, own side)
//   Gbar_l = D_l Ybar,  Ubar = sum_l (dG_l/dU)^T Gbar_l
// and, after the face phase turned the seeds into trace cotangents Tbar_f,
//   Qbar = V^T (Ubar + sum_f E_f^T Tbar_f).
// smem per block: bufA [5 nQ], bufG [15 nQ], bufC [5 nQ].

// Phase A.  rk == 0: Rbar given.  rk == 1 (one reverse LSERK stage):
// Kbar <- Kbar + b Qbar is the Rbar of this stage and Kbar <- a (Kbar + b Qbar)
// is written back.
template <bool CURVED>
__device__ __forceinline__ void element_vjp_a_t(const Ctx& c, const VjpArgs& va, int64_t s, double* bufA, double* bufG,
                                             double* bufC, int lane) {
  const TypeTab& T = c.tabs[c.slot_tab[s]];
  // curved element: pointwise metric, 1/J_q (hex) or the dense M_e^{-1}
  // (prism, pyramid) in place of the affine 1/J and diagonal M_ref^{-1}
  const double* cblk = CURVED ? c.cpool + c.slot_coff[s] : nullptr;
  const bool dense = CURVED && T.type != HEX;
  constexpr int nQ = knQ;
  const int nM = T.nM;
  const double* dp = c.dpool;
  const int64_t qoff = c.slot_qoff[s];
  constexpr int nQm = knQ;
  // forward nodal state and its traces (read by the face phase): kept by the
  // forward pass, or recomputed from Q
  if (va.stored) {
    const double* Un = c.Unod + c.slot_hoff[s];
    for (int w = lane; w < 5 * nQ; w += blockDim.x) bufA[w] = Un[w];
    __syncthreads();
  } else {
    for (int w = lane; w < 5 * nM; w += blockDim.x) bufC[w] = va.Q[qoff + w];
    __syncthreads();
    modal_to_nodal(c, T, bufC, bufA, bufG, lane);
    write_traces(c, T, s, bufA, c.T);
  }
  // scaled cotangent of the modal residual, rbar = M_e^{-1} Rbar (M_e symmetric)
  const double invJ = CURVED ? 1.0 : c.geo[s].invJ;
  double* rdst = dense ? bufC : bufG;   // bufC is free here (Q consumed above)
  for (int w = lane; w < 5 * nM; w += blockDim.x) {
    const int m = w % nM;
    double rb;
    if (va.rk) {
      rb = va.Kbar[qoff + w] + va.b * va.Qbar[qoff + w];
      va.Kbar[qoff + w] = va.a * rb;
    } else {
      rb = va.Rbar[qoff + w];
    }
    rdst[w] = dense ? rb : rb * dp[T.minv + m] * invJ;
  }
  __syncthreads();
  if (dense) {
    const double* Md = cblk + 11 * nQ;
    dense_product(Md, bufC, nM, [&](int m, double* acc) {
#pragma unroll
      for (int v = 0; v < 5; ++v) bufG[v * nM + m] = acc[v];
    });
    __syncthreads();
  }
  modal_to_nodal(c, T, bufG, bufC, bufG + 5 * nQm, lane);  // Ybar in bufC
  if (CURVED && !dense) {
    // curved hexahedron: the forward's diag(1/J_q) before V^T, transposed
    const double* iJ = cblk + 10 * nQ;
    for (int w = lane; w < 5 * nQ; w += blockDim.x) bufC[w] *= iJ[w % nQ];
    __syncthreads();
  }
  write_traces(c, T, s, bufC, c.Tv, 0x80000000u);          // seeds
  // Gbar_l = D_l Ybar (collocation derivative), D[i][i'] = Dt[i'][i]
  __syncthreads();
  fx_grad<kn>(bufC, bufG);
  // pointwise transpose of the contravariant flux
  {
    const ElemGeo& g = c.geo[s];
    double Jg[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) Jg[k] = g.Jg[k];
    double* Hb = c.H + c.slot_hoff[s];
    for (int q = lane; q < nQ; q += blockDim.x) {
      double U[5], Gb[3][5], Ub[5];
#pragma unroll
      for (int v = 0; v < 5; ++v) U[v] = bufA[v * nQ + q];
#pragma unroll
      for (int l = 0; l < 3; ++l)
#pragma unroll
        for (int v = 0; v < 5; ++v) Gb[l][v] = bufG[(l * 5 + v) * nQ + q];
      double M[3][3];
      if (CURVED) {
#pragma unroll
        for (int l = 0; l < 3; ++l)
#pragma unroll
          for (int d = 0; d < 3; ++d) M[l][d] = cblk[(l * 3 + d) * nQ + q];
      } else {
        point_metric(T.type, dp + T.wA + q * 9, Jg, M);
      }
      contravariant_vjp(U, M, c.gamma, Gb, Ub);
#pragma unroll
      for (int v = 0; v < 5; ++v) Hb[v * nQ + q] = Ub[v];
    }
  }
  __syncthreads();
}

template <bool ANY>
__device__ __forceinline__ void element_vjp_a(const Ctx& c, const VjpArgs& va, int64_t s, double* bufA, double* bufG,
                                              double* bufC, int lane) {
  if (ANY && c.slot_coff[s] >= 0) element_vjp_a_t<true>(c, va, s, bufA, bufG, bufC, lane);
  else element_vjp_a_t<false>(c, va, s, bufA, bufG, bufC, lane);
}

// Phase C: Qbar = V^T (Ubar + sum_f E_f^T Tbar_f); stored (rk == 0) or added
// with weight dt (rk == 1).
__device__ __forceinline__ void element_vjp_c(const Ctx& c, const VjpArgs& va, int64_t s, double* bufA, double* bufG,
                                           int lane) {
  const TypeTab& T = c.tabs[c.slot_tab[s]];
  Epilogue ep{va.rk ? Epilogue::kAxpy : Epilogue::kStore, false, va.rk ? va.dt : 1.0, va.Qbar + c.slot_qoff[s],
              nullptr, nullptr, nullptr, nullptr, 0.0, 0.0};
  element_backward<false>(c, T, s, bufA, bufG, lane, c.Tv, 0u, nullptr, ep);
}

// ------------------------------------------------------------------ Navier-Stokes adjoint element phases
//
// The forward state at Q is recomputed first (traces T, nodal state Unod,
// lifting values, gradient traces Vt and the nodal gradient DW).  Then:
//   A: Ybar = V diag(M_ref^-1 / J) Rbar, seeds -E_f Ybar (Tv), Fbar_l = D_l Ybar;
//      per point the transposed total flux F_e(U) - F_v(U, DW): Ubar -> H,
//      gradient cotangent -> DW (in place);
//   face flux adjoint: trace cotangents (Tv) and gradient-trace cotangents (Vtb);
//   B: DWbar_d = DW + sum_f E_f^T Vtb_f,d; Bbar_d = V (-1/J) M_ref^-1 V^T DWbar_d;
//      Lbar_f = -sum_d n_d(f) E_f Bbar_d (own side of L);
//      Wbar = sum_d sum_l M[l][d] D_l Bbar_d, Ubar += (dW/dU)^T Wbar (H);
//   lifting-value adjoint: trace cotangents += (dW/dU)^T of the face means (Tv);
//   C (shared with Euler): Qbar = V^T (Ubar + sum_f E_f^T Tbar_f).

// bufA += sum_f E_f^T faces_f, face values at (ft_mult ft[lf] + ft_add)
// (staged through bufS; bufX [5 nQ] scratch).
__device__ __forceinline__ void lift_add(const Ctx& c, const TypeTab& T, int64_t s, double* bufA, double* bufS,
                                      double* bufX, int lane, const double* faces, int ft_mult, int64_t ft_add) {
  const int nf = T.nfaces;
  const int64_t* ft = c.slot_ftoff + s * 6;
#pragma unroll
  for (int v = 0; v < 5; ++v)
    for (int w = lane; w < nf * kn2; w += blockDim.x) {
      const int lf = w / kn2, o = v * kn2 + w - lf * kn2;
      bufS[lf * 5 * kn2 + o] = faces[ft_mult * ft[lf] + ft_add + o];
    }
  __syncthreads();
  fx_lift<kn>(T, [&](int o) { return bufA[o]; }, bufS, 0u, bufX, [&](int o, double x) { bufA[o] = x; });
}

// Phase A (Navier-Stokes).  smem: bufY [5 nQ] | bufG [15 nQ] | bufS [5 nQ].
template <bool CURVED>
__device__ __forceinline__ void element_vjp_a_ns_t(const Ctx& c, const VjpArgs& va, int64_t s, double* smem, int lane) {
  const TypeTab& T = c.tabs[c.slot_tab[s]];
  constexpr int nQ = knQ;
  const int nM = T.nM;
  constexpr int nQm = knQ;
  double* bufY = smem;
  double* bufG = smem + 5 * nQm;
  double* bufS = smem + 20 * nQm;
  const double* dp = c.dpool;
  const int64_t qoff = c.slot_qoff[s];
  // curved element: dense M_e^{-1} (prism, pyramid) or 1/J_q (hex), pointwise metric
  const double* cblk = CURVED ? c.cpool + c.slot_coff[s] : nullptr;
  const bool dense = CURVED && T.type != HEX;
  const double invJ = CURVED ? 1.0 : c.geo[s].invJ;
  double* rdst = dense ? bufY : bufS;   // bufY is free until the modal -> nodal pass
  for (int w = lane; w < 5 * nM; w += blockDim.x) {
    const int m = w % nM;
    double rb;
    if (va.rk) {
      rb = va.Kbar[qoff + w] + va.b * va.Qbar[qoff + w];
      va.Kbar[qoff + w] = va.a * rb;
    } else {
      rb = va.Rbar[qoff + w];
    }
    rdst[w] = dense ? rb : rb * dp[T.minv + m] * invJ;
  }
  __syncthreads();
  if (dense) {
    const double* Md = cblk + 11 * nQ;
    dense_product(Md, bufY, nM, [&](int m, double* acc) {
#pragma unroll
      for (int v = 0; v < 5; ++v) bufS[v * nM + m] = acc[v];
    });
    __syncthreads();
  }
  modal_to_nodal(c, T, bufS, bufY, bufG, lane);
  if (CURVED && !dense) {
    const double* iJ = cblk + 10 * nQ;
    for (int w = lane; w < 5 * nQ; w += blockDim.x) bufY[w] *= iJ[w % nQ];
    __syncthreads();
  }
  write_traces(c, T, s, bufY, c.Tv, 0x80000000u);
  __syncthreads();
  fx_grad<kn>(bufY, bufG);
  {
    const ElemGeo& g = c.geo[s];
    double Jg[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) Jg[k] = g.Jg[k];
    const double gm1 = c.gamma - 1.0;
    const double* Un = c.Unod + c.slot_hoff[s];
    double* DWs = c.DW + 3 * c.slot_hoff[s];
    double* Hb = c.H + c.slot_hoff[s];
    for (int q = lane; q < nQ; q += blockDim.x) {
      double U[5], W[5], gr[15], Gb[3][5], Ub[5], Wb[5] = {0, 0, 0, 0, 0}, gb[15];
#pragma unroll
      for (int v = 0; v < 5; ++v) U[v] = Un[v * nQ + q];
#pragma unroll
      for (int t = 0; t < 15; ++t) {
        gr[t] = DWs[t * nQ + q];
        gb[t] = 0.0;
      }
#pragma unroll
      for (int l = 0; l < 3; ++l)
#pragma unroll
        for (int v = 0; v < 5; ++v) Gb[l][v] = bufG[(l * 5 + v) * nQ + q];
      double M[3][3];
      if (CURVED) {
#pragma unroll
        for (int l = 0; l < 3; ++l)
#pragma unroll
          for (int d = 0; d < 3; ++d) M[l][d] = cblk[(l * 3 + d) * nQ + q];
      } else {
        point_metric(T.type, dp + T.wA + q * 9, Jg, M);
      }
      contravariant_vjp(U, M, c.gamma, Gb, Ub);
      // G_l -= sum_d M[l][d] F_v[d]  =>  Fvbar[d] = -sum_l M[l][d] Gbar_l
      double Fvb[3][5];
#pragma unroll
      for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int v = 0; v < 5; ++v) Fvb[d][v] = -(M[0][d] * Gb[0][v] + M[1][d] * Gb[1][v] + M[2][d] * Gb[2][v]);
      primitive(U, gm1, W);
      viscous_flux_vjp(W, gr, c.mu, c.kappa, Fvb, Wb, gb);
      primitive_vjp(U, gm1, Wb, Ub);
#pragma unroll
      for (int v = 0; v < 5; ++v) Hb[v * nQ + q] = Ub[v];
#pragma unroll
      for (int t = 0; t < 15; ++t) DWs[t * nQ + q] = gb[t];
    }
  }
  __syncthreads();
}

// bufL_f -= n_d(f) E_f B on the element's own face points (bufL shared, [nf][5][n^2])
template <int n, bool CURVED>
__device__ __forceinline__ void lbar_traces_n(const Ctx& c, const TypeTab& T, int64_t s, const double* B, double* bufL,
                                           int d) {
  constexpr int n2 = n * n;
  const int64_t* ft = c.slot_ftoff + s * 6;
  fx_traces<n>(T, B, [&](int lf, int v, int p, double x) {
    const double nd = CURVED ? c.snrm[3 * (ft[lf] / 5) + d * n2 + p] : c.fnrm[(s * 6 + lf) * 3 + d];
    double* L = bufL + (lf * 5 + v) * n2 + p;
    *L = fma(-nd, x, *L);
  });
}

// Phase B (Navier-Stokes lifting transpose).
// smem: bufD [15 nQ] | bufB [5 nQ] | bufX [5 nQ] | bufW [5 nQ] | bufL [15 nQ].
template <bool CURVED>
__device__ __forceinline__ void element_vjp_b_ns_t(const Ctx& c, int64_t s, double* smem, int lane) {
  const TypeTab& T = c.tabs[c.slot_tab[s]];
  const double* cblk = CURVED ? c.cpool + c.slot_coff[s] : nullptr;
  constexpr int nQ = knQ, n2 = kn2;
  const int nf = T.nfaces;
  constexpr int nQm = knQ;
  double* bufD = smem;                 // smem + 15 nQm .. 20 nQm is scratch
  double* bufX = smem + 20 * nQm;
  double* bufW = smem + 25 * nQm;
  double* bufL = smem + 30 * nQm;
  const double* dp = c.dpool;
  const int64_t* ft = c.slot_ftoff + s * 6;
  const ElemGeo& g = c.geo[s];
  {
    const double* DWs = c.DW + 3 * c.slot_hoff[s];
    for (int w = lane; w < 15 * nQ; w += blockDim.x) bufD[w] = DWs[w];
  }
  __syncthreads();
  for (int d = 0; d < 3; ++d) lift_add(c, T, s, bufD + d * 5 * nQ, bufL, smem + 15 * nQm, lane, c.Vtb, 3, (int64_t)d * 5 * n2);
  for (int w = lane; w < 5 * nQ; w += blockDim.x) bufW[w] = 0.0;
  for (int w = lane; w < nf * 5 * n2; w += blockDim.x) bufL[w] = 0.0;
  __syncthreads();
  double Jg[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) Jg[k] = g.Jg[k];
  for (int d = 0; d < 3; ++d) {
    double* Bd = bufD + d * 5 * nQ;     // DWbar_d, replaced by Bbar_d
    if (T.type == HEX) {
      // V M^{-1} V^T = (W J)^{-1} (square V): pointwise
      const double* wq = dp + T.W;
      if (CURVED) {
        const double* iJ = cblk + 10 * nQ;
        for (int w = lane; w < 5 * nQ; w += blockDim.x) Bd[w] = -iJ[w % nQ] * Bd[w] * rcp(wq[w % nQ]);
      } else {
        for (int w = lane; w < 5 * nQ; w += blockDim.x) Bd[w] = -g.invJ * Bd[w] * rcp(wq[w % nQ]);
      }
      __syncthreads();
    } else {
      Epilogue ep{Epilogue::kStore, true, CURVED ? -1.0 : -g.invJ, bufX, nullptr, nullptr, nullptr, nullptr, 0.0, 0.0};
      if (CURVED) {
        ep.Md = cblk + 11 * nQ;        // symmetric: its own transpose
        ep.rbuf = smem + 15 * nQm;
      }
      nodal_to_modal<CURVED>(c, T, Bd, bufX, lane, ep);
      modal_to_nodal(c, T, bufX, Bd, bufX, lane);
    }
    // Lbar_f -= n_d(f) E_f Bbar_d on the own face points
    lbar_traces_n<kn, CURVED>(c, T, s, Bd, bufL, d);
    __syncthreads();
  }
  // Wbar = sum_d sum_l M[l][d] D_l Bbar_d = sum_k sum_{l: wA[l][k] != 0} wA[l][k] D_l C_k
  // with C_k = sum_d Jg[k][d] Bbar_d (in place of the Bbar_d); a curved
  // element takes the first form with its pointwise metric
  if (CURVED) {
    for (int d = 0; d < 3; ++d)
      for (int l = 0; l < 3; ++l) {
        fx_grad1<kn>(l, bufD + d * 5 * nQ, bufX);
        for (int w = lane; w < 5 * nQ; w += blockDim.x) bufW[w] = fma(cblk[(l * 3 + d) * nQ + w % nQ], bufX[w], bufW[w]);
        __syncthreads();
      }
  }
  for (int w = lane; w < (CURVED ? 0 : 5 * nQ); w += blockDim.x) {
    const double b0 = bufD[w], b1 = bufD[5 * nQ + w], b2 = bufD[10 * nQ + w];
#pragma unroll
    for (int kr = 0; kr < 3; ++kr)
      bufD[kr * 5 * nQ + w] = Jg[kr * 3] * b0 + Jg[kr * 3 + 1] * b1 + Jg[kr * 3 + 2] * b2;
  }
  __syncthreads();
  if (!CURVED) {
    const unsigned nz = kMetricMask[T.type];
    for (int kr = 0; kr < 3; ++kr)
      for (int l = 0; l < 3; ++l) {
        if (!((nz >> (3 * l + kr)) & 1u)) continue;
        fx_grad1<kn>(l, bufD + kr * 5 * nQ, bufX);
        for (int w = lane; w < 5 * nQ; w += blockDim.x) bufW[w] = fma(dp[T.wA + (w % nQ) * 9 + 3 * l + kr], bufX[w], bufW[w]);
        __syncthreads();
      }
  }
  __syncthreads();
  {
    const double gm1 = c.gamma - 1.0;
    const double* Un = c.Unod + c.slot_hoff[s];
    double* Hb = c.H + c.slot_hoff[s];
    for (int q = lane; q < nQ; q += blockDim.x) {
      double U[5], Wb[5], Ub[5] = {0, 0, 0, 0, 0};
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        U[v] = Un[v * nQ + q];
        Wb[v] = bufW[v * nQ + q];
      }
      primitive_vjp(U, gm1, Wb, Ub);
#pragma unroll
      for (int v = 0; v < 5; ++v) Hb[v * nQ + q] += Ub[v];
    }
    for (int w = lane; w < nf * 5 * n2; w += blockDim.x) {
      int lf = w / (5 * n2), r = w - lf * 5 * n2;
      c.L[ft[lf] + r] = bufL[w];
    }
  }
  __syncthreads();
}

template <bool ANY>
__device__ __forceinline__ void element_vjp_a_ns(const Ctx& c, const VjpArgs& va, int64_t s, double* smem, int lane) {
  if (ANY && c.slot_coff[s] >= 0) element_vjp_a_ns_t<true>(c, va, s, smem, lane);
  else element_vjp_a_ns_t<false>(c, va, s, smem, lane);
}

template <bool ANY>
__device__ __forceinline__ void element_vjp_b_ns(const Ctx& c, int64_t s, double* smem, int lane) {
  if (ANY && c.slot_coff[s] >= 0) element_vjp_b_ns_t<true>(c, s, smem, lane);
  else element_vjp_b_ns_t<false>(c, s, smem, lane);
}

// ------------------------------------------------------------------ kernels
//
// One block (1 to 4 warps) works on one element at a time; its threads share
// the element's shared-memory workspace bufA [5 nQ] + bufG [15 nQ].

// The launch's stage arguments with the state, register and time step taken
// from the device parameter block when the launch has one.
__device__ __forceinline__ StageArgs resolve_args(const StageArgs& a) {
  StageArgs r = a;
  if (a.dyn) {
    const RkDyn d = *a.dyn;
    r.Qin = d.Q;
    r.Qout = d.Q;
    r.K = d.K;
    r.dt = d.dt;
  }
  return r;
}

// One element per block (chunk_start null: the listed slots), or a persistent
// launch whose blocks pop chunks of the list from the queue.
template <int FAM, bool ANY, bool SPLIT>
__global__ void __launch_bounds__(128, FAM == kStage ? (SPLIT ? kSplitBlocks : kStageBlocks) : (FAM == kNs ? kNsBlocks : 1)) elem_kernel(const __grid_constant__ Ctx c, int mode,
                                                   const __grid_constant__ StageArgs io0,
                                                   const __grid_constant__ Sched sc) {
  extern __shared__ double smem[];
  __shared__ unsigned int s_chunk;
  const StageArgs io = resolve_args(io0);
  const int lane = threadIdx.x;
  double* bufA = smem;
  double* bufG = bufA + 5 * knQ;
  if (!sc.chunk_start) {
    const int64_t idx = blockIdx.x;
    if (idx >= sc.count) return;
    const int64_t s = sc.list ? sc.list[idx] : idx;
    if (c.tabs[c.slot_tab[s]].n == kn) process_element<FAM, ANY, SPLIT>(c, mode, io, s, bufA, bufG, lane);
    return;
  }
  // The previous launch on this stream used next_counter and has finished.
  if (blockIdx.x == 0 && threadIdx.x == 0 && sc.next_counter) *sc.next_counter = 0u;
  // Cost probe: time per element, summed per (type, N) table in shared bins
  // (thread 0 alone touches them) and flushed once at the end.
  __shared__ unsigned long long s_cost[2 * kMaxTabs];
  for (int t = lane; t < 2 * kMaxTabs; t += blockDim.x) s_cost[t] = 0ull;
  unsigned long long busy = 0;
  while (true) {
    if (lane == 0) s_chunk = atomicAdd(sc.counter, 1u);
    __syncthreads();
    const unsigned int ch = s_chunk;
    __syncthreads();
    if (ch >= sc.count) break;
    for (int64_t i = sc.chunk_start[ch]; i < sc.chunk_start[ch + 1]; ++i) {
      const int64_t s = sc.list ? sc.list[i] : i;
      const int tab = c.slot_tab[s];
      if (c.tabs[tab].n != kn) continue;   // a batch of several degrees: another launch's element
      uint64_t t0 = global_ns();
      process_element<FAM, ANY, SPLIT>(c, mode, io, s, bufA, bufG, lane);
      __syncthreads();
      uint64_t dtn = global_ns() - t0;
      if (lane == 0) {
        s_cost[2 * tab] += dtn;
        s_cost[2 * tab + 1] += 1ull;
      }
      busy += dtn;
    }
  }
  if (lane == 0 && c.cost) {
    for (int t = 0; t < kMaxTabs; ++t)
      if (s_cost[2 * t + 1]) {
        atomicAdd(c.cost + 2 * t, s_cost[2 * t]);
        atomicAdd(c.cost + 2 * t + 1, s_cost[2 * t + 1]);
      }
    if (busy) atomicAdd(c.sm_ns + smid(), busy);
  }
}

// ------------------------------------------------------------------ adjoint kernels

// One kernel per phase, so that each gets its own register allocation.
template <int PHASE, bool ANY>
__global__ void __launch_bounds__(128) elem_vjp_kernel(Ctx c, VjpArgs va) {
  extern __shared__ double smem[];
  const int64_t s = blockIdx.x;
  if (c.tabs[c.slot_tab[s]].n != kn) return;
  double* bufA = smem;
  double* bufG = bufA + 5 * knQ;
  double* bufC = bufG + 15 * knQ;
  if (PHASE == 0) element_vjp_a<ANY>(c, va, s, bufA, bufG, bufC, threadIdx.x);
  else if (PHASE == 10) element_vjp_a_ns<ANY>(c, va, s, smem, threadIdx.x);
  else if (PHASE == 11) element_vjp_b_ns<ANY>(c, s, smem, threadIdx.x);
  else element_vjp_c(c, va, s, bufA, bufG, threadIdx.x);
}

#if DG_PART == 1
// ------------------------------------------------------------------ moving meshes: stage mass matrices
//
// M^ = V^T diag(w J^) V with J^ = sum_k tau_k J_k per element (the stage
// value of J of a moving mesh).  Hexahedra hold s = W^{1/2} V q, so M^ q in
// their storage is J^ s pointwise and the solve a pointwise division.
// Prisms and pyramids: the product M^ x runs as the two sum-factorised
// transforms of the element kernel around the pointwise w J^ (FP64).  The
// solve is iterative refinement in FP64 around an FP32 Cholesky factor of the
// diagonally scaled S M^ S (S = diag(M^)^{-1/2}, condition number near
// max J / min J): x = 0, r = b; three times z = S (L L^T)^{-1} S r in FP32,
// x += z, r = b - M^ x in FP64.  Each FP32 solve gains about six digits,
// so the third correction leaves the FP64 rounding of M^ x.  Started from a
// nearby state x0 instead (the previous stage's, about 1e-3 away), two
// corrections reach the same.  FP64 work per solve is two products, against
// nM^3 / 3 FP64 flops for an FP64 Cholesky (FP64 issues at 1/64 of the FP32
// rate on this part).  A solve may keep its factor in global memory, and a
// later solve with a matrix equal to M^ within the FP32 rounding may use it
// instead of forming its own (the refinement runs with its own M^).
//
// smem: x, b, r [5][nM] and wJ [nQ] (FP64); bufA, bufB [5][nQ] (FP64,
// transforms; during the factor, bufA holds its two panel buffers); L
// (packed lower triangle), s, rdiag [nM] (FP32).  Block: 5 warps.
constexpr int kMassThreads = 160;
static_assert(kMassThreads % 32 == 0 && kMassThreads >= 64, "the factor needs warp 0 and at least one other warp");
constexpr int kMassRows = 4;   // rows per lane in the warp solves: nM <= 128
constexpr int kMassBlocks2 = 6, kMassBlocks = 5;   // resident blocks per SM (two rows per lane, more)

// the FP32 factor is kept packed: row i of the lower triangle at i (i + 1) / 2
__host__ __device__ __forceinline__ int lro(int i) { return i * (i + 1) / 2; }

__host__ __device__ __forceinline__ size_t mass_smem_doubles(int nM, int nQ) {
  return 15 * (size_t)nM + (size_t)nQ + 10 * (size_t)nQ;
}

// r = b - M^ x (or r = M^ x when b is null); tid = threadIdx.x
__device__ void mass_product(const Ctx& c, const TypeTab& T, const double* x, const double* wJ, const double* b,
                             double* r, double* bufA, double* bufB, int tid) {
  constexpr int nQ = knQ;
  const int nM = T.nM;
  modal_to_nodal_passes<false>(c, T, x, bufA, bufB);
  for (int w = tid; w < 5 * nQ; w += blockDim.x) bufA[w] *= wJ[w % nQ];
  __syncthreads();
  Epilogue ep{Epilogue::kStore, false, 1.0, r, nullptr, nullptr, nullptr, nullptr, 0.0, 0.0};
  nodal_to_modal_t<false>(c, T, bufA, bufB, tid, ep);
  if (b) {
    for (int w = tid; w < 5 * nM; w += blockDim.x) r[w] = b[w] - r[w];
    __syncthreads();
  }
}

// x += S (L L^T)^{-1} S r: warp v solves for variable v (ROWS rows per lane
// in registers, one shuffle per pivot, the rows already solved masked by a
// zero coefficient instead of a branch).  The five warps run side by side.
template <int ROWS>
__device__ void mass_correct_t(const float* L, const float* sc, const float* rdiag, const double* r, double* x,
                               int nM) {
  const int v = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (v < 5) {
    const double* rv = r + v * nM;
    float y[ROWS], sl[ROWS];
#pragma unroll
    for (int m = 0; m < ROWS; ++m) {
      const int i = lane + 32 * m;
      sl[m] = i < nM ? sc[min(i, nM - 1)] : 0.0f;
      y[m] = i < nM ? sl[m] * (float)rv[min(i, nM - 1)] : 0.0f;
    }
    // L y = S r
#pragma unroll
    for (int m = 0; m < ROWS; ++m) {
      const int jend = min(32, nM - 32 * m);
      for (int jj = 0; jj < jend; ++jj) {
        const int j = 32 * m + jj;
        const float yj = __shfl_sync(0xffffffffu, y[m], jj) * rdiag[j];
        y[m] = lane == jj ? yj : y[m];
#pragma unroll
        for (int m2 = m; m2 < ROWS; ++m2) {
          const int i = lane + 32 * m2;
          const float lij = (i > j && i < nM) ? L[lro(min(i, nM - 1)) + j] : 0.0f;
          y[m2] = fmaf(-lij, yj, y[m2]);
        }
      }
    }
    // L^T z = y
#pragma unroll
    for (int m = ROWS - 1; m >= 0; --m) {
      const int jend = min(32, nM - 32 * m);
      for (int jj = jend - 1; jj >= 0; --jj) {
        const int j = 32 * m + jj;
        const float zj = __shfl_sync(0xffffffffu, y[m], jj) * rdiag[j];
        y[m] = lane == jj ? zj : y[m];
#pragma unroll
        for (int m2 = 0; m2 <= m; ++m2) {
          const int i = lane + 32 * m2;
          const float lji = i < j ? L[lro(j) + min(i, j)] : 0.0f;
          y[m2] = fmaf(-lji, zj, y[m2]);
        }
      }
    }
    double* xv = x + v * nM;
#pragma unroll
    for (int m = 0; m < ROWS; ++m) {
      const int i = lane + 32 * m;
      if (i < nM) xv[i] += (double)(sl[m] * y[m]);
    }
  }
  __syncthreads();
}

// The FP32 factor L L^T = S M^ S of one element (S = diag(M^)^{-1/2}), from
// the four packed FP32 coefficient triangles Mk and the powers f of the
// stage time; pan: two buffers of four floats per row on a 16-byte boundary
// (scratch).
// One warp: columns jh .. jh+3 of the FP32 factor (rows jh .. nM-1, by lane
// in registers).  With prev (the previous panel's rows, four values each),
// its rank-4 update of these columns comes first (the earlier panels' updates
// are in L already).  Leaves the factored columns in L, their reciprocal
// diagonal in rdiag and the rows below the panel in out.
template <int ROWS>
__device__ __forceinline__ void mass_panel(float* L, float* rdiag, float4* out, const float4* prev, int jh, int nM,
                                           int lane) {
  const int hw = min(4, nM - jh);
  float p[ROWS][4];
#pragma unroll
  for (int m = 0; m < ROWS; ++m) {
    const int i = jh + lane + 32 * m, ic = min(i, nM - 1);
#pragma unroll
    for (int cc = 0; cc < 4; ++cc)
      p[m][cc] = (i < nM && cc < hw && jh + cc <= i) ? L[lro(ic) + min(jh + cc, ic)] : 0.0f;
  }
  if (prev) {
#pragma unroll
    for (int m = 0; m < ROWS; ++m) {
      const float4 a = prev[min(jh + lane + 32 * m, nM - 1)];
#pragma unroll
      for (int cc = 0; cc < 4; ++cc) {
        const float4 bb = prev[min(jh + cc, nM - 1)];
        p[m][cc] = fmaf(-a.w, bb.w, fmaf(-a.z, bb.z, fmaf(-a.y, bb.y, fmaf(-a.x, bb.x, p[m][cc]))));
      }
    }
  }
#pragma unroll
  for (int cc = 0; cc < 4; ++cc) {
    if (cc < hw) {
      // row jh + cc is lane cc of the first register row
      const float rd = rsqrtf(__shfl_sync(0xffffffffu, p[0][cc], cc));
      if (lane == 0) rdiag[jh + cc] = rd;
#pragma unroll
      for (int m = 0; m < ROWS; ++m)
        if (lane + 32 * m > cc) p[m][cc] *= rd;
#pragma unroll
      for (int c2 = cc + 1; c2 < 4; ++c2) {
        const float l = __shfl_sync(0xffffffffu, p[0][cc], c2);
#pragma unroll
        for (int m = 0; m < ROWS; ++m) p[m][c2] = fmaf(-p[m][cc], l, p[m][c2]);
      }
    }
  }
#pragma unroll
  for (int m = 0; m < ROWS; ++m) {
    const int i = jh + lane + 32 * m;
    if (i < nM) {
#pragma unroll
      for (int cc = 0; cc < 4; ++cc)
        if (cc < hw && jh + cc < i) L[lro(i) + jh + cc] = p[m][cc];
      if (i >= jh + hw)
        out[i] = make_float4(p[m][0], hw > 1 ? p[m][1] : 0.0f, hw > 2 ? p[m][2] : 0.0f, hw > 3 ? p[m][3] : 0.0f);
    }
  }
}

template <int ROWS>
__device__ void mass_factor(const float* Mk, float f0, float f1, float f2, float f3, float* L, float* sc, float* rdiag,
                            float4* pan, int nM) {
  const int tid = threadIdx.x, bd = blockDim.x, lane = tid & 31, warp = tid >> 5, nwarps = bd >> 5;
  const int np = lro(nM);
  // FP32 S M^ S from the FP32 coefficients, all four kept packed (lower
  // triangle, the layout of L): contiguous loads, then the scaling in
  // shared memory
#pragma unroll 4
  for (int u = tid; u < np; u += bd)
    L[u] = fmaf(f3, Mk[3 * np + u], fmaf(f2, Mk[2 * np + u], fmaf(f1, Mk[np + u], f0 * Mk[u])));
  __syncthreads();
  for (int a = tid; a < nM; a += bd) sc[a] = rsqrtf(L[lro(a) + a]);
  __syncthreads();
  for (int a = warp; a < nM; a += nwarps) {
    const float sa = sc[a];
    for (int k = lane; k <= a; k += 32) L[lro(a) + k] *= sa * sc[k];
  }
  __syncthreads();
  // right-looking Cholesky in panels of four columns with one panel of
  // lookahead: while warps 1-4 apply the current panel's rank-4 update to the
  // trailing lower triangle beyond the next panel (four rows per warp at a
  // time, independent chains that share each column's load), warp 0 applies
  // it to the next panel's four columns in registers and factors them.  One
  // barrier per panel.  L's diagonal is kept as its reciprocal in rdiag.
  float4* cur = pan;
  float4* nxt = pan + nM;
  if (warp == 0) mass_panel<ROWS>(L, rdiag, cur, nullptr, 0, nM, lane);
  __syncthreads();
  for (int j0 = 0; j0 + 4 < nM; j0 += 4) {
    const int jt = j0 + 4;   // the next panel
    if (warp == 0) {
      mass_panel<ROWS>(L, rdiag, nxt, cur, jt, nM, lane);
    } else {
      const int j4 = jt + 4, wt = warp - 1, nwt = nwarps - 1;
      for (int i = j4 + wt; i < nM; i += 4 * nwt) {
        float4 lr[4];
        int last = i;
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          lr[g] = cur[min(i + g * nwt, nM - 1)];
          if (i + g * nwt < nM) last = i + g * nwt;
        }
        for (int k = j4 + lane; k <= last; k += 32) {
          const float4 ck = cur[k];
          float v[4];
#pragma unroll
          for (int g = 0; g < 4; ++g) {
            const int ig = i + g * nwt;
            v[g] = (ig < nM && k <= ig) ? L[lro(min(ig, nM - 1)) + k] : 0.0f;
          }
#pragma unroll
          for (int g = 0; g < 4; ++g)
            v[g] = fmaf(-lr[g].w, ck.w, fmaf(-lr[g].z, ck.z, fmaf(-lr[g].y, ck.y, fmaf(-lr[g].x, ck.x, v[g]))));
#pragma unroll
          for (int g = 0; g < 4; ++g) {
            const int ig = i + g * nwt;
            if (ig < nM && k <= ig) L[lro(ig) + k] = v[g];
          }
        }
      }
    }
    __syncthreads();
    float4* t = cur;
    cur = nxt;
    nxt = t;
  }
}

template <int ROWS, int MINB>
__global__ void __launch_bounds__(kMassThreads, MINB) moving_mass_kernel(Ctx c, const int64_t* list, int64_t E,
                                                                   const double* in, double* out, const double* x0,
                                                                   double t0, double t1, double t2, double t3,
                                                                   int weight, int max_nM, int max_nQ, int nblk,
                                                                   int64_t blk_stride, float* fac_out,
                                                                   const float* fac_in) {
  extern __shared__ double sm[];
  const int tid = threadIdx.x, bd = blockDim.x;
  double* x = sm;
  double* b = x + 5 * max_nM;
  double* r = b + 5 * max_nM;
  double* wJ = r + 5 * max_nM;
  double* bufA = wJ + max_nQ;
  double* bufB = bufA + 5 * max_nQ;
  float* L = reinterpret_cast<float*>(bufB + 5 * max_nQ);
  float* sc = L + lro(max_nM);
  float* rdiag = sc + max_nM;
  for (int64_t e = blockIdx.x; e < E; e += gridDim.x) {
    const int64_t s = list[e];
    const TypeTab& T = c.tabs[c.slot_tab[s]];
    constexpr int nQ = knQ;
    const int nM = T.nM;
    const int64_t qoff = c.slot_qoff[s];
    const double* m = c.mpool + c.slot_moff[s];
    if (T.type == HEX) {
      for (int w = tid; w < 5 * nQ * nblk; w += bd) {
        const int kb = w / (5 * nQ), wl = w - kb * 5 * nQ, q = wl % nQ;
        const int64_t o = qoff + kb * blk_stride + wl;
        const double J = fma(t3, m[30 * nQ + q], fma(t2, m[29 * nQ + q], fma(t1, m[28 * nQ + q], t0 * m[27 * nQ + q])));
        const double v = in[o];
        out[o] = weight ? v * J : v / J;
      }
      continue;   // block-uniform branch, no shared memory used
    }
    const double* W = c.dpool + T.W;
    for (int q = tid; q < nQ; q += bd)
      wJ[q] = W[q] * fma(t3, m[30 * nQ + q], fma(t2, m[29 * nQ + q], fma(t1, m[28 * nQ + q], t0 * m[27 * nQ + q])));
    for (int w = tid; w < 5 * nM; w += bd) b[w] = in[qoff + w];
    __syncthreads();
    if (weight) {
      mass_product(c, T, b, wJ, nullptr, r, bufA, bufB, tid);
      for (int w = tid; w < 5 * nM; w += bd) out[qoff + w] = r[w];
      __syncthreads();
      continue;
    }
    const int np = lro(nM);
    if (fac_in) {
      // a factor kept from a solve with (nearly) the same matrix: the
      // refinement below corrects for the difference in FP64
      const float* F = fac_in + c.slot_mmoff[s];
      for (int u = tid; u < np; u += bd) L[u] = F[u];
      for (int a = tid; a < nM; a += bd) {
        sc[a] = F[np + a];
        rdiag[a] = F[np + nM + a];
      }
      __syncthreads();
    } else {
      // pan lives in the transform buffer, idle until the first product, on
      // a 16-byte boundary
      mass_factor<ROWS>(c.mk32 + c.slot_mmoff[s], (float)t0, (float)t1, (float)t2, (float)t3, L, sc, rdiag,
                  reinterpret_cast<float4*>(bufA + ((15 * max_nM + max_nQ) & 1)), nM);
      if (fac_out) {
        // kept for a later solve (the lifting of the stage): [L][s][rdiag]
        float* F = fac_out + c.slot_mmoff[s];
        for (int u = tid; u < np; u += bd) F[u] = L[u];
        for (int a = tid; a < nM; a += bd) {
          F[np + a] = sc[a];
          F[np + nM + a] = rdiag[a];
        }
      }
    }
    // every block of five variables with the one factor (nblk > 1: the
    // lifting's three directions), from x0 (a nearby solution: one
    // correction fewer) or from zero
    for (int kb = 0; kb < nblk; ++kb) {
      const int64_t o = qoff + kb * blk_stride;
      if (kb > 0) {
        for (int w = tid; w < 5 * nM; w += bd) b[w] = in[o + w];
        __syncthreads();
      }
      for (int w = tid; w < 5 * nM; w += bd) {
        x[w] = x0 ? x0[o + w] : 0.0;
        r[w] = b[w];
      }
      __syncthreads();
      if (x0) mass_product(c, T, x, wJ, b, r, bufA, bufB, tid);
      const int ncorr = x0 ? 2 : 3;
      for (int it = 0; it < ncorr; ++it) {
        mass_correct_t<ROWS>(L, sc, rdiag, r, x, nM);
        if (it + 1 < ncorr) mass_product(c, T, x, wJ, b, r, bufA, bufB, tid);
      }
      for (int w = tid; w < 5 * nM; w += bd) out[o + w] = x[w];
      __syncthreads();
    }
  }
}
#endif  // DG_PART == 1

}  // namespace

namespace {

template <class K>
cudaError_t set_smem(K kernel, int bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

constexpr int kD = (int)sizeof(double);
constexpr int kStageBytes = 20 * knQ * kD, kNsBytes = (20 * knQ + kNsG) * kD;
// the split form's workspace: bufA [5 nQ] + two-point quantities [kTP][nQ] +
// face states [kTP][6 n^2] + one direction's pair fluxes [n^2][n(n-1)/2][5]
// and face-state fluxes [n^2][2 n][5]
constexpr int kSplitWork = (5 * knQ + kTP * knQ + kTP * 6 * kn2 + kn2 * (kn * (kn - 1) / 2) * 5 + kn2 * 2 * kn * 5) * kD;
constexpr int kSplitBytes = kStageBytes > kSplitWork ? kStageBytes : kSplitWork;

template <int FAM, bool ANY, bool SPLIT>
void launch_family(const Ctx& c, int mode, const StageArgs& a, const Sched& s, bool balanced, int grid, int wpb,
                   int bytes, cudaStream_t st) {
  Sched sc = s;
  if (!balanced) {
    if (s.count <= 0) return;
    sc.chunk_start = nullptr;
    grid = (int)s.count;
  }
  elem_kernel<FAM, ANY, SPLIT><<<(unsigned)grid, 32 * wpb, bytes, st>>>(c, mode, a, sc);
}

#if DG_PART == 0
void element(const Ctx& c, int mode, const StageArgs& a, const Sched& s, bool balanced, int grid, int wpb,
             cudaStream_t st) {
  if (c.slot_coff) launch_family<kStage, true, false>(c, mode, a, s, balanced, grid, wpb, kStageBytes, st);
  else if (c.split) launch_family<kStage, false, true>(c, mode, a, s, balanced, grid, wpb, kSplitBytes, st);
  else launch_family<kStage, false, false>(c, mode, a, s, balanced, grid, wpb, kStageBytes, st);
}

cudaError_t attributes(int wpb, int* blocks_per_sm, bool curved, bool split) {
  cudaError_t e;
  if ((e = set_smem(elem_kernel<kStage, false, false>, kStageBytes)) != cudaSuccess) return e;
  if ((e = set_smem(elem_kernel<kStage, true, false>, kStageBytes)) != cudaSuccess) return e;
  if ((e = set_smem(elem_kernel<kStage, false, true>, kSplitBytes)) != cudaSuccess) return e;
  if (curved)
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, elem_kernel<kStage, true, false>, 32 * wpb,
                                                         kStageBytes);
  if (split)
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, elem_kernel<kStage, false, true>, 32 * wpb,
                                                         kSplitBytes);
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, elem_kernel<kStage, false, false>, 32 * wpb,
                                                       kStageBytes);
}
#elif DG_PART == 1
void element(const Ctx& c, int mode, const StageArgs& a, const Sched& s, bool balanced, int grid, int wpb,
             cudaStream_t st) {
  // one-shot maps; kGather / kScatter: one block per listed hexahedron
  if (mode != kNsVolume) launch_family<kMisc, true, false>(c, mode, a, s, balanced, grid, wpb, kStageBytes, st);
  else if (c.slot_coff) launch_family<kNs, true, false>(c, mode, a, s, balanced, grid, wpb, kNsBytes, st);
  else launch_family<kNs, false, false>(c, mode, a, s, balanced, grid, wpb, kNsBytes, st);
}

cudaError_t attributes(int wpb, int* blocks_per_sm, bool curved, bool) {
  cudaError_t e;
  if ((e = set_smem(elem_kernel<kMisc, true, false>, kStageBytes)) != cudaSuccess) return e;
  if ((e = set_smem(elem_kernel<kNs, false, false>, kNsBytes)) != cudaSuccess) return e;
  if ((e = set_smem(elem_kernel<kNs, true, false>, kNsBytes)) != cudaSuccess) return e;
  if (curved)
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, elem_kernel<kNs, true, false>, 32 * wpb,
                                                         kNsBytes);
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, elem_kernel<kNs, false, false>, 32 * wpb,
                                                       kNsBytes);
}

cudaError_t mass(const Ctx& c, const int64_t* list, int64_t n_slots, const double* in, double* out, const double* x0,
                 const double* tau, int weight, int max_nM, int max_nQ, int grid, cudaStream_t st, int nblk,
                 int64_t blk_stride, float* fac_out, const float* fac_in) {
  if (weight && nblk != 1) return cudaErrorInvalidValue;
  if (weight && (fac_out || fac_in)) return cudaErrorInvalidValue;
  if (max_nM > 32 * kMassRows) return cudaErrorInvalidValue;
  size_t bytes = 0;
  if (max_nM > 0)
    bytes = sizeof(double) * mass_smem_doubles(max_nM, max_nQ) + sizeof(float) * ((size_t)lro(max_nM) + 2 * (size_t)max_nM);
  auto launch = [&](auto kern) -> cudaError_t {
    if (bytes > 48 * 1024) {
      cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
      if (e != cudaSuccess) return e;
    }
    kern<<<grid, kMassThreads, bytes, st>>>(c, list, n_slots, in, out, x0, tau[0], tau[1], tau[2], tau[3], weight,
                                             max_nM, max_nQ, nblk, blk_stride, fac_out, fac_in);
    return cudaSuccess;
  };
  // rows per lane in the warp solves and the panel (nM <= 32 ROWS): two up to
  // N = 3 and for pyramids of N = 4, three for prisms of N = 4 and pyramids of
  // N = 5, four for prisms of N = 5 (moving prisms and pyramids end there).
  // Hexahedra (max_nM = 0, pointwise, every N) run in the degree's smallest.
  cudaError_t e = cudaErrorInvalidValue;
  if constexpr (kn == 6) {
    if (max_nM <= 64) e = launch(moving_mass_kernel<3, kMassBlocks>);
  } else {
    if (max_nM <= (kn <= 5 ? 64 : 0)) e = launch(moving_mass_kernel<2, kMassBlocks2>);
  }
  if constexpr (kn == 5 || kn == 6)
    if (max_nM > 64 && max_nM <= 96) e = launch(moving_mass_kernel<3, kMassBlocks>);
  if constexpr (kn == 6)
    if (max_nM > 96) e = launch(moving_mass_kernel<4, kMassBlocks>);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}
#else
template <bool ANY>
void vjp_t(const Ctx& c, int phase, const VjpArgs& va, unsigned nb, int nt, cudaStream_t st) {
  switch (phase) {
    case 0: elem_vjp_kernel<0, ANY><<<nb, nt, 25 * knQ * kD, st>>>(c, va); break;
    case 10: elem_vjp_kernel<10, ANY><<<nb, nt, 25 * knQ * kD, st>>>(c, va); break;
    case 11: elem_vjp_kernel<11, ANY><<<nb, nt, 45 * knQ * kD, st>>>(c, va); break;
    default: elem_vjp_kernel<2, false><<<nb, nt, 20 * knQ * kD, st>>>(c, va); break;   // phase C has no geometry
  }
}

void vjp(const Ctx& c, int phase, const VjpArgs& va, int64_t nelem, int wpb, cudaStream_t st) {
  if (nelem <= 0) return;
  if (c.slot_coff) vjp_t<true>(c, phase, va, (unsigned)nelem, 32 * wpb, st);
  else vjp_t<false>(c, phase, va, (unsigned)nelem, 32 * wpb, st);
}

template <bool ANY>
cudaError_t vjp_attributes() {
  cudaError_t e;
  if ((e = set_smem(elem_vjp_kernel<0, ANY>, 25 * knQ * kD)) != cudaSuccess) return e;
  if ((e = set_smem(elem_vjp_kernel<2, false>, 20 * knQ * kD)) != cudaSuccess) return e;
  if ((e = set_smem(elem_vjp_kernel<10, ANY>, 25 * knQ * kD)) != cudaSuccess) return e;
  return set_smem(elem_vjp_kernel<11, ANY>, 45 * knQ * kD);
}

cudaError_t attributes(int, int*, bool, bool) {
  cudaError_t e = vjp_attributes<false>();
  return e != cudaSuccess ? e : vjp_attributes<true>();
}
#endif

}  // namespace

#define DG_OPS_NAME3(n, p) elem_ops_##n##_##p
#define DG_OPS_NAME2(n, p) DG_OPS_NAME3(n, p)
#define DG_OPS_NAME DG_OPS_NAME2(DG_N, DG_PART)
extern const ElemOps DG_OPS_NAME;
#if DG_PART == 0
const ElemOps DG_OPS_NAME = {element, nullptr, nullptr, attributes};
#elif DG_PART == 1
const ElemOps DG_OPS_NAME = {element, nullptr, mass, attributes};
#else
const ElemOps DG_OPS_NAME = {nullptr, vjp, nullptr, attributes};
#endif

}  // namespace dgk
