// The FP64 face flux: traces interpolated in block fixed point (dg_fixed.cuh)
// and the pointwise HLL and central stress fluxes in floating point, written for
// few FP64 instructions.  Included by dg_kernels.cuh.
//
// Bound by the FP64 pipe (83 % busy): about 96 operations a face point in 2D (175 with
// floating-point interpolation, IEEE division and square root and FP64
// comparisons); comparisons, minima and maxima run on the integer pipe, the
// reciprocal and roots start from the FP32 unit (dg_math64.cuh).  524,288
// triangles, p = 2: 1060 -> 587 us, p = 1: 474 -> 305 us; 8,192 triangles,
// p = 2: 24.7 -> 20.6 us; 200 intervals: 10.3 -> 8.3 us.
#pragma once

namespace dgswe {

// Symmetric-gradient components the stress needs: du/dx, or (d11, d22, d12).
template <int DIM>
constexpr int sym_comps() { return DIM == 1 ? 1 : 3; }

// One side of a face point: HLL ingredients and the stress row.
template <int DIM>
struct Side64 {
  double un, c;         // normal velocity, wave speed
  double h, q, p;       // depth, normal discharge, g_c h^2
  double m, t[DIM];     // -(Q . n)_j / 2 = m t_j
};
template <int DIM>
__device__ __forceinline__ void side64(const double* V, const double* d, const double* n, const Phys<double>& ph,
                                       Side64<DIM>& s) {
  const double h = V[0];
  double un = V[1] * n[0];
  if constexpr (DIM == 2) un += V[2] * n[1];
  const double gh = ph.gc * h;
  s.un = un;
  s.c = sqrt_pos(max_pos(gh, ph.gc * ph.h_floor));
  s.h = h;
  s.q = h * un;
  s.p = h * gh;
  if constexpr (DIM == 1) {
    s.m = stress_mu1<double>(d[0], ph) * ((-0.5 * ph.rho_inv) * h);
    s.t[0] = (2.0 * d[0]) * n[0];
  } else {
    // a_i = d_ii + tr D; d11 a_1 + d22 a_2 = d11^2 + d22^2 + tr^2
    const double a1 = fma(2.0, d[0], d[1]), a2 = fma(2.0, d[1], d[0]);
    const double s2 = fma(0.5, fma(d[0], a1, d[1] * a2), d[2] * d[2]);
    s.m = stress_mu2<double>(s2, ph) * ((-0.5 * ph.rho_inv) * h);
    s.t[0] = a1 * n[0] + d[2] * n[1];
    s.t[1] = d[2] * n[0] + a2 * n[1];
  }
}

// Weighted numerical flux of one point: HLL for F minus the central flux of Q.
// With F = x F_a + y F_b + z (U_b - U_a) and F = u q + n p / 2 per side, the
// momentum flux is A u_a + B u_b + n (x p_a + y p_b) / 2 with A = x q_a - z h_a,
// B = y q_b + z h_b: 16 operations with the depth flux instead of 24 (upwind: x
// or y = 1, the rest 0).  The depth flux keeps the difference of the depths: it
// is small against c h in slow flow, A + B would round at c h.
template <int DIM>
__device__ __forceinline__ void flux64(const double* Vm, const double* Vp, const double* dm, const double* dp,
                                       const double* n, const Phys<double>& ph, double w, double* out) {
  Side64<DIM> a, b;
  side64<DIM>(Vm, dm, n, ph, a);
  side64<DIM>(Vp, dp, n, ph, b);
  const double SL = min_f64(a.un - a.c, b.un - b.c), SR = max_f64(a.un + a.c, b.un + b.c);
  double F0 = a.q, A = a.q, B = 0.0, P = a.p;
  if (__double2hiint(SL) < 0) {
    if (__double2hiint(SR) < 0) {
      A = 0.0;
      F0 = B = b.q;
      P = b.p;
    } else {
      const double inv = rcp_pos(SR - SL);
      const double x = SR * inv, y = -SL * inv, z = SL * x;
      A = fma(x, a.q, -z * a.h);
      B = fma(y, b.q, z * b.h);
      P = fma(x, a.p, y * b.p);
      F0 = fma(x, a.q, fma(y, b.q, z * (b.h - a.h)));
    }
  }
  out[0] = w * F0;
  const double Ph = 0.5 * P;
#pragma unroll
  for (int j = 0; j < DIM; ++j)
    out[1 + j] = w * fma(A, Vm[1 + j], fma(B, Vp[1 + j], fma(Ph, n[j], fma(a.m, a.t[j], b.m * b.t[j]))));
}

// Traces of one side of a face at its nodes, as operands with one exponent per
// field: h, u, then the symmetric-gradient components.
template <int DIM, int P>
struct Trace64 {
  static constexpr int NX = DIM + 1 + sym_comps<DIM>();
  Fx x[NX][Sh<DIM, P>::NFP];
  int e[NX];  // exponent of the unit: results of a table with scale cs are r 2^(e - cs)
};
template <int DIM, int P, bool COH>
__device__ __forceinline__ void load_trace64(const double* __restrict__ V, const double* __restrict__ E, size_t KN,
                                             size_t eo, const int8_t* fm, bool flip, Trace64<DIM, P>& t) {
  using S = Sh<DIM, P>;
  constexpr int NFP = S::NFP, NV = S::NV;
  size_t at[NFP];
#pragma unroll
  for (int k = 0; k < NFP; ++k) at[k] = eo + fm[flip ? NFP - 1 - k : k];
#pragma unroll
  for (int v = 0; v < NV + 2; ++v) {  // h, u, d11, d22
    const double* src = v < NV ? V + v * KN : E + (v == NV ? 0 : 3) * KN;
    double x[NFP];
    int e = 0;
#pragma unroll
    for (int k = 0; k < NFP; ++k) {
      x[k] = DG_LDC(COH, src, at[k]);
      e = max(e, fx_exp(x[k]));
    }
#pragma unroll
    for (int k = 0; k < NFP; ++k) t.x[v][k] = fx_from<5>(x[k], e);
    t.e[v] = e - 1024;
  }
  {  // d12 = (E_12 + E_21) / 2
    double x[NFP], y[NFP];
    int e = 0;
#pragma unroll
    for (int k = 0; k < NFP; ++k) {
      x[k] = DG_LDC(COH, E, KN + at[k]);
      y[k] = DG_LDC(COH, E, 2 * KN + at[k]);
      e = max(e, max(fx_exp(x[k]), fx_exp(y[k])));
    }
#pragma unroll
    for (int k = 0; k < NFP; ++k) {
      const Fx p = fx_from<4>(x[k], e), q = fx_from<4>(y[k], e);
      t.x[NV + 2][k] = Fx{p.h + q.h, p.l + q.l};
    }
    t.e[NV + 2] = e - 1024;  // (one for the format, less one for the half)
  }
}
template <int DIM, int P>
__device__ __forceinline__ void trace_at(const Trace64<DIM, P>& t, const FaceOps<DIM, P, double>& ops, int m,
                                         double* V, double* d) {
  using S = Sh<DIM, P>;
  constexpr int NFP = S::NFP, NV = S::NV;
#pragma unroll
  for (int v = 0; v < Trace64<DIM, P>::NX; ++v) {
    FxAcc s{0, 0};
#pragma unroll
    for (int k = 0; k < NFP; ++k) fx_mac(s, t.x[v][k], ops.Lfx[m * NFP + k]);
    const double r = fx_to(fx_sum(s), fx_scale(t.e[v] - ops.cs, t.e[v] <= kFxMaxExp - 1024));
    if (v < NV) V[v] = r;
    else d[v - NV] = r;
  }
}

// Face fc: its points m0 .. m1 - 1 (all of them, or one).
template <int DIM, int P, bool COH>
__device__ __forceinline__ void face_fx(int fc, int m0, int m1, int e1, int f1, int e2, int f2, const double (&n)[DIM],
                                        double wsj, int K, int F, const double* __restrict__ V,
                                        const double* __restrict__ E, double* __restrict__ wflux,
                                        const FaceOps<DIM, P, double>& ops, const Phys<double>& ph,
                                        const BCEntry<double>* __restrict__ bct) {
  using S = Sh<DIM, P>;
  constexpr int NP = S::NP, NFP = S::NFP, NFQ = S::NFQ, NV = S::NV, ND = sym_comps<DIM>();
  const size_t KN = (size_t)K * NP, FQ = (size_t)F * NFQ;
  const bool interior = e2 >= 0;
  if constexpr (DIM == 1) {
    // one node, one point: no interpolation
    double Vm[NV], Vp[NV], dm[ND], dp[ND], out[NV];
    const size_t a = (size_t)e1 * NP + ops.fmask[f1], b = interior ? (size_t)e2 * NP + ops.fmask[f2] : a;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      Vm[v] = DG_LDC(COH, V, v * KN + a);
      Vp[v] = DG_LDC(COH, V, v * KN + b);
    }
    dm[0] = DG_LDC(COH, E, a);
    dp[0] = DG_LDC(COH, E, b);
    if (!interior) {
      const BCEntry<double> bc = bct[-1 - e2];
      ghost_V<DIM, double>(Vm, n, bc, Vp);
      ghost_E<DIM, double>(dm, bc, dp);
    }
    flux64<DIM>(Vm, Vp, dm, dp, n, ph, ops.wf[0] * wsj, out);
#pragma unroll
    for (int v = 0; v < NV; ++v) wflux[v * FQ + fc] = out[v];
  } else {
    Trace64<DIM, P> tm, tp;
    load_trace64<DIM, P, COH>(V, E, KN, (size_t)e1 * NP, ops.fmask + f1 * NFP, false, tm);
    if (interior) load_trace64<DIM, P, COH>(V, E, KN, (size_t)e2 * NP, ops.fmask + f2 * NFP, true, tp);
#pragma unroll 1
    for (int m = m0; m < m1; ++m) {
      double Vm[NV], Vp[NV], dm[ND], dp[ND], out[NV];
      trace_at<DIM, P>(tm, ops, m, Vm, dm);
      if (interior) {
        trace_at<DIM, P>(tp, ops, m, Vp, dp);
      } else {
        const BCEntry<double> bc = bct[-1 - e2];
        ghost_V<DIM, double>(Vm, n, bc, Vp);
        dp[0] = bc.mode[3] == 1 ? bc.val[3] : dm[0];
        dp[1] = bc.mode[6] == 1 ? bc.val[6] : dm[1];
        dp[2] = dm[2];
        if (bc.mode[4] == 1 || bc.mode[5] == 1) {
          // a prescribed E_12 or E_21: the two components apart
          double x = 0.0, y = 0.0;
          for (int k = 0; k < NFP; ++k) {
            const size_t a = (size_t)e1 * NP + ops.fmask[f1 * NFP + k];
            x += ops.Lf[m * NFP + k] * DG_LDC(COH, E, KN + a);
            y += ops.Lf[m * NFP + k] * DG_LDC(COH, E, 2 * KN + a);
          }
          dp[2] = 0.5 * ((bc.mode[4] == 1 ? bc.val[4] : x) + (bc.mode[5] == 1 ? bc.val[5] : y));
        }
      }
      flux64<DIM>(Vm, Vp, dm, dp, n, ph, ops.wf[m] * wsj, out);
#pragma unroll
      for (int v = 0; v < NV; ++v) wflux[v * FQ + (size_t)fc * NFQ + m] = out[v];
    }
  }
}

}  // namespace dgswe
