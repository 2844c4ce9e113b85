// Face kernels (Riemann and viscous fluxes, their adjoints) and the layout copies.
#include <algorithm>

#include "dg_physics.cuh"

namespace dgk {

namespace {

template <bool CURVED>
__global__ void face_kernel(Ctx c) {
  extern __shared__ double sF[];
  const FaceBlock fb = c.fblocks[blockIdx.x];
  const int n = fb.n, n2 = n * n, items = fb.count * n2;
  const double gamma = c.gamma;
  for (int w = threadIdx.x; w < items; w += blockDim.x) {
    int fl = w / n2, p = w - fl * n2;
    const FaceRec& R = c.faces[fb.first + fl];
    const double* T0 = c.T + R.toff;
    const double* T1 = T0 + 5 * n2;
    double UL[5], UR[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) UL[v] = T0[v * n2 + p];
    if (R.map >= 0) {
      int j = c.perms[(size_t)R.map + p];
#pragma unroll
      for (int v = 0; v < 5; ++v) UR[v] = T1[v * n2 + j];
    } else {
      const double* D = c.dense + (size_t)(-1 - R.map) + (size_t)p * n2;
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        double acc = 0.0;
        for (int j = 0; j < n2; ++j) acc = fma(D[j], T1[v * n2 + j], acc);
        UR[v] = acc;
      }
    }
    double nrm[3] = {R.nrm[0], R.nrm[1], R.nrm[2]};
    const bool cg = CURVED && R.cgeo >= 0;
    if (cg) {
      // curved owner: the normal at this point
      const double* G = c.fgeo + R.cgeo;
      nrm[0] = G[p];
      nrm[1] = G[n2 + p];
      nrm[2] = G[2 * n2 + p];
    }
    const double wS = cg ? c.fgeo[R.cgeo + 3 * n2 + p] : c.dpool[c.tabs[R.owner_tab].fw + R.owner_lf * n2 + p] * R.S;
    double Fs[5];
    if (CURVED && c.fmot && cg) {
      // moving mesh (LF only): the normal mesh speed at the owner's point
      const double* xf = c.fmot + 3 * (int64_t)R.cgeo + 9 * n2 + p;
      const double sn = nrm[0] * xf[0] + nrm[1] * xf[n2] + nrm[2] * xf[2 * n2];
      flux_lf_moving_scaled(UL, UR, nrm, wS, sn, gamma, Fs);
    } else if (c.flux == 0) {
      flux_lf_scaled(UL, UR, nrm, wS, gamma, Fs);   // wS F*
    } else if (c.flux == 2) {
      // entropy-conservative: Chandrashekar's F# contracted with wS n
      double PL[kTP], PR[kTP];
      two_point_state(UL, gamma - 1.0, PL);
      two_point_state(UR, gamma - 1.0, PR);
      const double m[3] = {wS * nrm[0], wS * nrm[1], wS * nrm[2]};
      two_point_flux(PL, 1, PR, 1, m, 1.0 / (gamma - 1.0), Fs);
    } else {
      flux_roe(UL, UR, nrm, gamma, Fs);
#pragma unroll
      for (int v = 0; v < 5; ++v) Fs[v] *= wS;
    }
    if (R.map >= 0) {
      // permutation map: this thread alone read T0[p] and T1[perm[p]], so it
      // writes both results in place at once
      const int j = c.perms[(size_t)R.map + p];
      double* W0 = c.T + R.toff;
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        W0[v * n2 + p] = Fs[v];
        W0[(5 + v) * n2 + j] = -Fs[v];
      }
    } else {
#pragma unroll
      for (int v = 0; v < 5; ++v) sF[(fl * 5 + v) * n2 + p] = Fs[v];
    }
  }
  __syncthreads();
  // interpolating maps: the neighbour's share needs every owner point first
  for (int w = threadIdx.x; w < items; w += blockDim.x) {
    int fl = w / n2, q = w - fl * n2;
    const FaceRec& R = c.faces[fb.first + fl];
    if (R.map >= 0) continue;
    double* T0 = c.T + R.toff;
    double* T1 = T0 + 5 * n2;
    const double* F = sF + fl * 5 * n2;
#pragma unroll
    for (int v = 0; v < 5; ++v) T0[v * n2 + q] = F[v * n2 + q];
    {
      const double* D = c.dense + (size_t)(-1 - R.map) + q;
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        double acc = 0.0;
        for (int p = 0; p < n2; ++p) acc = fma(D[(size_t)p * n2], F[v * n2 + p], acc);
        T1[v * n2 + q] = -acc;
      }
    }
  }
}

// Navier-Stokes face phases.  KIND 0 (BR1 lifting): per owner point p,
// W* = (W(U-) + W(U+))/2 with U+ the neighbour trace mapped to the owner's
// points, and L = w S W* (owner side) / Map^T (w S W*) (neighbour side); the
// element multiplies by its own outward normal.  KIND 1 (flux): the inviscid
// Riemann flux minus the central viscous flux (F_v(U-, g-) + F_v(U+, g+)).n/2,
// g the lifted gradient traces, times w S, written over the traces as in the
// Euler face kernel.
template <int KIND, bool CURVED>
__global__ void face_ns_kernel(Ctx c) {
  extern __shared__ double sF[];
  const FaceBlock fb = c.fblocks[blockIdx.x];
  const int n = fb.n, n2 = n * n, items = fb.count * n2;
  const double gamma = c.gamma, gm1 = gamma - 1.0;
  for (int w = threadIdx.x; w < items; w += blockDim.x) {
    int fl = w / n2, p = w - fl * n2;
    const FaceRec& R = c.faces[fb.first + fl];
    const double* T0 = c.T + R.toff;
    const double* T1 = T0 + 5 * n2;
    double UL[5], UR[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) UL[v] = T0[v * n2 + p];
    if (R.map >= 0) {
      int j = c.perms[(size_t)R.map + p];
#pragma unroll
      for (int v = 0; v < 5; ++v) UR[v] = T1[v * n2 + j];
    } else {
      const double* D = c.dense + (size_t)(-1 - R.map) + (size_t)p * n2;
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        double acc = 0.0;
        for (int j = 0; j < n2; ++j) acc = fma(D[j], T1[v * n2 + j], acc);
        UR[v] = acc;
      }
    }
    const bool cg = CURVED && R.cgeo >= 0;   // curved owner: per-point normal and w S
    const double wS = cg ? c.fgeo[R.cgeo + 3 * n2 + p] : c.dpool[c.tabs[R.owner_tab].fw + R.owner_lf * n2 + p] * R.S;
    double Fs[5];   // w S times the value
    if (KIND == 0) {
      double WL[5], WR[5];
      primitive(UL, gm1, WL);
      primitive(UR, gm1, WR);
      const double h = 0.5 * wS;
#pragma unroll
      for (int v = 0; v < 5; ++v) Fs[v] = h * (WL[v] + WR[v]);
    } else {
      double nrm[3] = {R.nrm[0], R.nrm[1], R.nrm[2]};
      if (cg) {
        nrm[0] = c.fgeo[R.cgeo + p];
        nrm[1] = c.fgeo[R.cgeo + n2 + p];
        nrm[2] = c.fgeo[R.cgeo + 2 * n2 + p];
      }
      // everything with the scaled normal s = (w S / 2) n: the inviscid flux as
      // in flux_lf_scaled, the viscous one as the sum of both sides' F_v.s
      const double h = 0.5 * wS;
      const double s[3] = {h * nrm[0], h * nrm[1], h * nrm[2]};
      double rL, pL, rR, pR;
      if (c.flux == 0) {
        LfSide L, Q;
        if (CURVED && c.fmot && cg) {
          // moving mesh: the LF flux in the frame of the normal mesh speed
          const double* xf = c.fmot + 3 * (int64_t)R.cgeo + 9 * n2 + p;
          const double sig = s[0] * xf[0] + s[1] * xf[n2] + s[2] * xf[2 * n2];
          lf_side<true>(UL, s, h, sig, gm1, gamma, L);
          lf_side<true>(UR, s, h, sig, gm1, gamma, Q);
          lf_combine_moving(UL, UR, s, sig, L, Q, Fs);
        } else {
          lf_side<false>(UL, s, h, 0.0, gm1, gamma, L);
          lf_side<false>(UR, s, h, 0.0, gm1, gamma, Q);
          lf_combine(UL, UR, s, L, Q, Fs);
        }
        rL = L.r;
        pL = L.p;
        rR = Q.r;
        pR = Q.p;
      } else {
        flux_roe(UL, UR, nrm, gamma, Fs);
#pragma unroll
        for (int v = 0; v < 5; ++v) Fs[v] *= wS;
        double W[5];
        primitive(UL, gm1, W);
        rL = rcp(UL[0]);
        pL = W[4];
        primitive(UR, gm1, W);
        rR = rcp(UR[0]);
        pR = W[4];
      }
      const double* V0 = c.Vt + 3 * R.toff;
      const double* V1 = V0 + 15 * n2;
      double g[15], u[3], q[4];
#pragma unroll
      for (int t = 0; t < 15; ++t) g[t] = V0[t * n2 + p];
#pragma unroll
      for (int d = 0; d < 3; ++d) u[d] = UL[1 + d] * rL;
      viscous_flux_normal(rL, u, pL, g, s, c.mu, c.kappa, q);
#pragma unroll
      for (int v = 0; v < 4; ++v) Fs[1 + v] -= q[v];
      if (R.map >= 0) {
        int j = c.perms[(size_t)R.map + p];
#pragma unroll
        for (int t = 0; t < 15; ++t) g[t] = V1[t * n2 + j];
      } else {
        const double* D = c.dense + (size_t)(-1 - R.map) + (size_t)p * n2;
#pragma unroll
        for (int t = 0; t < 15; ++t) {
          double acc = 0.0;
          for (int j = 0; j < n2; ++j) acc = fma(D[j], V1[t * n2 + j], acc);
          g[t] = acc;
        }
      }
#pragma unroll
      for (int d = 0; d < 3; ++d) u[d] = UR[1 + d] * rR;
      viscous_flux_normal(rR, u, pR, g, s, c.mu, c.kappa, q);
#pragma unroll
      for (int v = 0; v < 4; ++v) Fs[1 + v] -= q[v];
    }
    if (R.map >= 0) {
      // permutation map: direct writes (this thread alone read the inputs at
      // p and perm[p]; the flux kind overwrites them in place)
      const int j = c.perms[(size_t)R.map + p];
      double* O0 = (KIND == 0 ? c.L : c.T) + R.toff;
      const double nb = KIND == 0 ? 1.0 : -1.0;
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        O0[v * n2 + p] = Fs[v];
        O0[(5 + v) * n2 + j] = nb * Fs[v];
      }
    } else {
#pragma unroll
      for (int v = 0; v < 5; ++v) sF[(fl * 5 + v) * n2 + p] = Fs[v];
    }
  }
  __syncthreads();
  double* out = KIND == 0 ? c.L : c.T;
  const double nb_sign = KIND == 0 ? 1.0 : -1.0;
  for (int w = threadIdx.x; w < items; w += blockDim.x) {
    int fl = w / n2, q = w - fl * n2;
    const FaceRec& R = c.faces[fb.first + fl];
    if (R.map >= 0) continue;
    double* O0 = out + R.toff;
    double* O1 = O0 + 5 * n2;
    const double* F = sF + fl * 5 * n2;
#pragma unroll
    for (int v = 0; v < 5; ++v) O0[v * n2 + q] = F[v * n2 + q];
    {
      const double* D = c.dense + (size_t)(-1 - R.map) + q;
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        double acc = 0.0;
        for (int p = 0; p < n2; ++p) acc = fma(D[(size_t)p * n2], F[v * n2 + p], acc);
        O1[v * n2 + q] = nb_sign * acc;
      }
    }
  }
}

// Face phase of the adjoint.  Per owner face point p, with Map the
// neighbour -> owner point map of the forward face phase:
//   g(p) = wS_p (seed_own(p) - (Map seed_nb)(p))     (cotangent of F*)
//   (Tbar-, Tbar+) = (dF*/dU-, dF*/dU+)^T g
//   Tbar_own = Tbar-,  Tbar_nb = Map^T Tbar+        (written over the seeds)
template <bool CURVED>
__global__ void face_vjp_kernel(Ctx c) {
  extern __shared__ double sF[];
  const FaceBlock fb = c.fblocks[blockIdx.x];
  const int n = fb.n, n2 = n * n, items = fb.count * n2;
  double* sR = sF + 32 * 5 * n2;
  const double gamma = c.gamma;
  for (int w = threadIdx.x; w < items; w += blockDim.x) {
    int fl = w / n2, p = w - fl * n2;
    const FaceRec& R = c.faces[fb.first + fl];
    const double* T0 = c.T + R.toff;
    const double* T1 = T0 + 5 * n2;
    const double* S0 = c.Tv + R.toff;
    const double* S1 = S0 + 5 * n2;
    double UL[5], UR[5], g[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      UL[v] = T0[v * n2 + p];
      g[v] = S0[v * n2 + p];
    }
    if (R.map >= 0) {
      int j = c.perms[(size_t)R.map + p];
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        UR[v] = T1[v * n2 + j];
        g[v] -= S1[v * n2 + j];
      }
    } else {
      const double* D = c.dense + (size_t)(-1 - R.map) + (size_t)p * n2;
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        double a = 0.0, b = 0.0;
        for (int j = 0; j < n2; ++j) {
          a = fma(D[j], T1[v * n2 + j], a);
          b = fma(D[j], S1[v * n2 + j], b);
        }
        UR[v] = a;
        g[v] -= b;
      }
    }
    const bool cg = CURVED && R.cgeo >= 0;
    const double wS = cg ? c.fgeo[R.cgeo + 3 * n2 + p]
                         : c.dpool[c.tabs[R.owner_tab].fw + R.owner_lf * n2 + p] * R.S;
#pragma unroll
    for (int v = 0; v < 5; ++v) g[v] *= wS;
    double nrm[3] = {R.nrm[0], R.nrm[1], R.nrm[2]};
    if (cg) {
      const double* G = c.fgeo + R.cgeo;
      nrm[0] = G[p];
      nrm[1] = G[n2 + p];
      nrm[2] = G[2 * n2 + p];
    }
    double UbL[5] = {0, 0, 0, 0, 0}, UbR[5] = {0, 0, 0, 0, 0};
    if (c.flux == 0) flux_lf_vjp(UL, UR, nrm, gamma, g, UbL, UbR);
    else flux_roe_vjp(UL, UR, nrm, gamma, g, UbL, UbR);
    if (R.map >= 0) {
      // permutation map: this thread alone read the seeds at p and perm[p]
      const int j = c.perms[(size_t)R.map + p];
      double* W0 = c.Tv + R.toff;
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        W0[v * n2 + p] = UbL[v];
        W0[(5 + v) * n2 + j] = UbR[v];
      }
    } else {
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        sF[(fl * 5 + v) * n2 + p] = UbL[v];
        sR[(fl * 5 + v) * n2 + p] = UbR[v];
      }
    }
  }
  __syncthreads();
  for (int w = threadIdx.x; w < items; w += blockDim.x) {
    int fl = w / n2, q = w - fl * n2;
    const FaceRec& R = c.faces[fb.first + fl];
    if (R.map >= 0) continue;
    double* S0 = c.Tv + R.toff;
    double* S1 = S0 + 5 * n2;
    const double* Fl = sF + fl * 5 * n2;
    const double* Fr = sR + fl * 5 * n2;
#pragma unroll
    for (int v = 0; v < 5; ++v) S0[v * n2 + q] = Fl[v * n2 + q];
    {
      const double* D = c.dense + (size_t)(-1 - R.map) + q;
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        double acc = 0.0;
        for (int p = 0; p < n2; ++p) acc = fma(D[(size_t)p * n2], Fr[v * n2 + p], acc);
        S1[v * n2 + q] = acc;
      }
    }
  }
}

// Navier-Stokes face adjoints.
// KIND 1 (flux): g = wS (seed_own - Map seed_nb) is the cotangent of the
//   unscaled flux F* = Riemann(U-, U+) - (F_v(U-, g-) + F_v(U+, g+)).n/2;
//   trace cotangents Tv (own side: Ubar-, neighbour: Map^T Ubar+) and
//   gradient-trace cotangents Vtb (likewise).  Faces with a permutation map
//   are finished by the thread that owns the point (it alone read the inputs
//   at p and perm[p]); on interpolating faces the neighbour's gradient
//   cotangent at the owner's points is parked in the owner half of Vt (read
//   only by the same thread) and the transposed map runs after a barrier.
// KIND 0 (lifting values): Wbar = wS (Lbar_own + Map Lbar_nb) / 2 for both
//   means' arguments; Tv += (dW/dU)^T Wbar (own), Map^T (neighbour).
// At most 7 warps (n <= 7) per block; two resident blocks at the largest n
// (three at n = 5) instead of the two that 168 registers allow.
template <int KIND, bool CURVED>
__global__ void __launch_bounds__(224, 2) face_ns_vjp_kernel(Ctx c) {
  extern __shared__ double sF[];
  const FaceBlock fb = c.fblocks[blockIdx.x];
  const int n = fb.n, n2 = n * n, items = fb.count * n2;
  double* sR = sF + 32 * 5 * n2;
  const double gamma = c.gamma, gm1 = gamma - 1.0;
  for (int w = threadIdx.x; w < items; w += blockDim.x) {
    int fl = w / n2, p = w - fl * n2;
    const FaceRec& R = c.faces[fb.first + fl];
    const double* T0 = c.T + R.toff;
    const double* T1 = T0 + 5 * n2;
    const double* S0 = (KIND == 1 ? c.Tv : c.L) + R.toff;
    const double* S1 = S0 + 5 * n2;
    double UL[5], UR[5], gs[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      UL[v] = T0[v * n2 + p];
      gs[v] = S0[v * n2 + p];
    }
    const double sgn = KIND == 1 ? -1.0 : 1.0;
    if (R.map >= 0) {
      int j = c.perms[(size_t)R.map + p];
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        UR[v] = T1[v * n2 + j];
        gs[v] += sgn * S1[v * n2 + j];
      }
    } else {
      const double* D = c.dense + (size_t)(-1 - R.map) + (size_t)p * n2;
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        double a = 0.0, b = 0.0;
        for (int j = 0; j < n2; ++j) {
          a = fma(D[j], T1[v * n2 + j], a);
          b = fma(D[j], S1[v * n2 + j], b);
        }
        UR[v] = a;
        gs[v] += sgn * b;
      }
    }
    const bool cg = CURVED && R.cgeo >= 0;   // curved owner: per-point normal and w S
    const double wS = cg ? c.fgeo[R.cgeo + 3 * n2 + p] : c.dpool[c.tabs[R.owner_tab].fw + R.owner_lf * n2 + p] * R.S;
    double UbL[5] = {0, 0, 0, 0, 0}, UbR[5] = {0, 0, 0, 0, 0};
    if (KIND == 0) {
      double Wb[5];
#pragma unroll
      for (int v = 0; v < 5; ++v) Wb[v] = 0.5 * wS * gs[v];
      primitive_vjp(UL, gm1, Wb, UbL);
      primitive_vjp(UR, gm1, Wb, UbR);
    } else {
#pragma unroll
      for (int v = 0; v < 5; ++v) gs[v] *= wS;
      double nrm[3] = {R.nrm[0], R.nrm[1], R.nrm[2]};
      if (cg) {
        nrm[0] = c.fgeo[R.cgeo + p];
        nrm[1] = c.fgeo[R.cgeo + n2 + p];
        nrm[2] = c.fgeo[R.cgeo + 2 * n2 + p];
      }
      if (c.flux == 0) flux_lf_vjp(UL, UR, nrm, gamma, gs, UbL, UbR);
      else flux_roe_vjp(UL, UR, nrm, gamma, gs, UbL, UbR);
      double Fvb[3][5];
#pragma unroll
      for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int v = 0; v < 5; ++v) Fvb[d][v] = -0.5 * nrm[d] * gs[v];
      double* V0 = c.Vt + 3 * R.toff;
      const double* V1 = V0 + 15 * n2;
      double gr[15], gb[15], W[5], Wb[5];
      // owner side
#pragma unroll
      for (int t = 0; t < 15; ++t) {
        gr[t] = V0[t * n2 + p];
        gb[t] = 0.0;
      }
#pragma unroll
      for (int v = 0; v < 5; ++v) Wb[v] = 0.0;
      primitive(UL, gm1, W);
      viscous_flux_vjp(W, gr, c.mu, c.kappa, Fvb, Wb, gb);
      primitive_vjp(UL, gm1, Wb, UbL);
      double* B0 = c.Vtb + 3 * R.toff;
#pragma unroll
      for (int t = 0; t < 15; ++t) B0[t * n2 + p] = gb[t];
      // neighbour side at the owner's points
      if (R.map >= 0) {
        int j = c.perms[(size_t)R.map + p];
#pragma unroll
        for (int t = 0; t < 15; ++t) gr[t] = V1[t * n2 + j];
      } else {
        const double* D = c.dense + (size_t)(-1 - R.map) + (size_t)p * n2;
#pragma unroll
        for (int t = 0; t < 15; ++t) {
          double acc = 0.0;
          for (int j = 0; j < n2; ++j) acc = fma(D[j], V1[t * n2 + j], acc);
          gr[t] = acc;
        }
      }
#pragma unroll
      for (int t = 0; t < 15; ++t) gb[t] = 0.0;
#pragma unroll
      for (int v = 0; v < 5; ++v) Wb[v] = 0.0;
      primitive(UR, gm1, W);
      viscous_flux_vjp(W, gr, c.mu, c.kappa, Fvb, Wb, gb);
      primitive_vjp(UR, gm1, Wb, UbR);
      if (R.map >= 0) {
        const int j = c.perms[(size_t)R.map + p];
        double* B1 = B0 + 15 * n2;
#pragma unroll
        for (int t = 0; t < 15; ++t) B1[t * n2 + j] = gb[t];
      } else {
#pragma unroll
        for (int t = 0; t < 15; ++t) V0[t * n2 + p] = gb[t];
      }
    }
    if (R.map >= 0) {
      // permutation map: this thread alone read the inputs at p and perm[p]
      const int j = c.perms[(size_t)R.map + p];
      double* W0 = c.Tv + R.toff;
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        if (KIND == 0) {
          W0[v * n2 + p] += UbL[v];
          W0[(5 + v) * n2 + j] += UbR[v];
        } else {
          W0[v * n2 + p] = UbL[v];
          W0[(5 + v) * n2 + j] = UbR[v];
        }
      }
    } else {
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        sF[(fl * 5 + v) * n2 + p] = UbL[v];
        sR[(fl * 5 + v) * n2 + p] = UbR[v];
      }
    }
  }
  __syncthreads();
  for (int w = threadIdx.x; w < items; w += blockDim.x) {
    int fl = w / n2, q = w - fl * n2;
    const FaceRec& R = c.faces[fb.first + fl];
    if (R.map >= 0) continue;
    double* S0 = c.Tv + R.toff;
    double* S1 = S0 + 5 * n2;
    const double* Fl = sF + fl * 5 * n2;
    const double* Fr = sR + fl * 5 * n2;
    const double keep = KIND == 0 ? 1.0 : 0.0;     // lifting values add to the flux cotangents
#pragma unroll
    for (int v = 0; v < 5; ++v) S0[v * n2 + q] = keep * S0[v * n2 + q] + Fl[v * n2 + q];
    const double* P0 = c.Vt + 3 * R.toff;          // parked neighbour gradient cotangents
    double* B1 = c.Vtb + 3 * R.toff + 15 * n2;
    {
      const double* D = c.dense + (size_t)(-1 - R.map) + q;
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        double acc = 0.0;
        for (int p = 0; p < n2; ++p) acc = fma(D[(size_t)p * n2], Fr[v * n2 + p], acc);
        S1[v * n2 + q] = keep * S1[v * n2 + q] + acc;
      }
      if (KIND == 1) {
        for (int t = 0; t < 15; ++t) {
          double acc = 0.0;
          for (int p = 0; p < n2; ++p) acc = fma(D[(size_t)p * n2], P0[t * n2 + p], acc);
          B1[t * n2 + q] = acc;
        }
      }
    }
  }
}

// Storage <-> caller layout copies (warp per element).
// Halo exchange of a partition mesh: copies whole face-side trace blocks of
// `per` doubles between the face buffer at the listed offsets and a packed
// buffer (pack: buffer block k <- T[off[k]]; unpack: T[off[k]] <- block k).
__global__ void halo_copy_kernel(const double* __restrict__ src, double* __restrict__ dst,
                                 const int64_t* __restrict__ off, int64_t count, int per, int pack, int mult) {
  for (int64_t k = blockIdx.x; k < count; k += gridDim.x) {
    const int64_t o = mult * off[k];
    for (int w = threadIdx.x; w < per; w += blockDim.x) {
      if (pack) dst[k * per + w] = src[o + w];
      else dst[o + w] = src[k * per + w];
    }
  }
}

__global__ void rk_params_kernel(RkDyn* d, double* Q, double* K, double dt) {
  d->Q = Q;
  d->K = K;
  d->dt = dt;
}

__global__ void permute_kernel(Ctx c, const double* __restrict__ src, double* __restrict__ dst, int64_t E, int to_storage) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int64_t s = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp;
  if (s >= E) return;
  const int nM = c.tabs[c.slot_tab[s]].nM;
  int64_t so = c.slot_qoff[s], eo = c.elem_qoff[c.elem_of_slot[s]];
  const double* a = src + (to_storage ? eo : so);
  double* b = dst + (to_storage ? so : eo);
  for (int w = lane; w < 5 * nM; w += 32) b[w] = a[w];
}

}  // namespace

namespace {
template <class K>
cudaError_t set_smem(K kernel, int bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}
}  // namespace

int face_block_threads(int n) { return 32 * n; }

// The shared-memory limits are per kernel function and process-wide, so they
// are set for the largest face any mesh may hold (N = kMaxN).
cudaError_t face_kernel_attributes() {
  cudaError_t e;
  const int fbytes = 32 * 5 * kMaxn * kMaxn * (int)sizeof(double);
  if ((e = set_smem(face_ns_kernel<0, false>, fbytes)) != cudaSuccess) return e;
  if ((e = set_smem(face_ns_kernel<1, false>, fbytes)) != cudaSuccess) return e;
  if ((e = set_smem(face_ns_kernel<0, true>, fbytes)) != cudaSuccess) return e;
  if ((e = set_smem(face_ns_kernel<1, true>, fbytes)) != cudaSuccess) return e;
  if ((e = set_smem(face_ns_vjp_kernel<0, false>, 2 * fbytes)) != cudaSuccess) return e;
  if ((e = set_smem(face_ns_vjp_kernel<1, false>, 2 * fbytes)) != cudaSuccess) return e;
  if ((e = set_smem(face_ns_vjp_kernel<0, true>, 2 * fbytes)) != cudaSuccess) return e;
  if ((e = set_smem(face_ns_vjp_kernel<1, true>, 2 * fbytes)) != cudaSuccess) return e;
  if ((e = set_smem(face_kernel<false>, fbytes)) != cudaSuccess) return e;
  if ((e = set_smem(face_kernel<true>, fbytes)) != cudaSuccess) return e;
  if ((e = set_smem(face_vjp_kernel<false>, 2 * fbytes)) != cudaSuccess) return e;
  return set_smem(face_vjp_kernel<true>, 2 * fbytes);
}

void launch_faces_ns_vjp(const Ctx& c, int64_t nblocks, int n, int kind, cudaStream_t st) {
  if (nblocks <= 0) return;
  int bytes = 2 * 32 * 5 * n * n * (int)sizeof(double);
  const unsigned nb = (unsigned)nblocks, nt = face_block_threads(n);
  if (c.fgeo) {
    if (kind == 0) face_ns_vjp_kernel<0, true><<<nb, nt, bytes, st>>>(c);
    else face_ns_vjp_kernel<1, true><<<nb, nt, bytes, st>>>(c);
  } else {
    if (kind == 0) face_ns_vjp_kernel<0, false><<<nb, nt, bytes, st>>>(c);
    else face_ns_vjp_kernel<1, false><<<nb, nt, bytes, st>>>(c);
  }
}

void launch_faces_vjp(const Ctx& c, int64_t nblocks, int n, cudaStream_t st) {
  if (nblocks <= 0) return;
  int bytes = 2 * 32 * 5 * n * n * (int)sizeof(double);
  if (c.fgeo) face_vjp_kernel<true><<<(unsigned)nblocks, face_block_threads(n), bytes, st>>>(c);
  else face_vjp_kernel<false><<<(unsigned)nblocks, face_block_threads(n), bytes, st>>>(c);
}

void launch_faces_ns(const Ctx& c, int64_t nblocks, int n, int kind, cudaStream_t st) {
  if (nblocks <= 0) return;
  int bytes = 32 * 5 * n * n * (int)sizeof(double);
  const unsigned nb = (unsigned)nblocks, nt = face_block_threads(n);
  if (c.fgeo) {
    if (kind == 0) face_ns_kernel<0, true><<<nb, nt, bytes, st>>>(c);
    else face_ns_kernel<1, true><<<nb, nt, bytes, st>>>(c);
  } else {
    if (kind == 0) face_ns_kernel<0, false><<<nb, nt, bytes, st>>>(c);
    else face_ns_kernel<1, false><<<nb, nt, bytes, st>>>(c);
  }
}

void launch_faces(const Ctx& c, int64_t nblocks, int n, cudaStream_t st) {
  if (nblocks <= 0) return;
  int bytes = 32 * 5 * n * n * (int)sizeof(double);
  if (c.fgeo) face_kernel<true><<<(unsigned)nblocks, face_block_threads(n), bytes, st>>>(c);
  else face_kernel<false><<<(unsigned)nblocks, face_block_threads(n), bytes, st>>>(c);
}

void launch_halo_copy(const double* src, double* dst, const int64_t* off, int64_t count, int per, bool pack,
                      cudaStream_t st, int mult) {
  if (count <= 0) return;
  const unsigned blocks = (unsigned)std::min<int64_t>(count, 65535);
  halo_copy_kernel<<<blocks, 128, 0, st>>>(src, dst, off, count, per, pack ? 1 : 0, mult);
}

void launch_rk_params(RkDyn* d, double* Q, double* K, double dt, cudaStream_t st) {
  rk_params_kernel<<<1, 1, 0, st>>>(d, Q, K, dt);
}

void rk_params_node(cudaKernelNodeParams* p, void** args) {
  p->func = (void*)rk_params_kernel;
  p->gridDim = dim3(1, 1, 1);
  p->blockDim = dim3(1, 1, 1);
  p->sharedMemBytes = 0;
  p->kernelParams = args;
  p->extra = nullptr;
}

bool is_rk_params_kernel(const void* func) { return func == (const void*)rk_params_kernel; }

void launch_permute(const Ctx& c, const double* src, double* dst, int64_t E, int to_storage, cudaStream_t st) {
  const int wpb = 4;
  int64_t blocks = (E + wpb - 1) / wpb;
  permute_kernel<<<(unsigned)blocks, 32 * wpb, 0, st>>>(c, src, dst, E, to_storage);
}

}  // namespace dgk
