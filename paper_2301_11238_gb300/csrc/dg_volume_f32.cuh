// The FP32 volume pass of one element in packed arithmetic.  Included by
// dg_kernels.cuh.
//
// fma.rn.f32x2 does two multiply-adds in one instruction (58.7 of them a clock
// and SM measured, 117 multiply-adds; the scalar FFMA 91), so the contractions
// run on pairs of neighbouring nodes: an interpolation is NP / 2 packed
// multiply-adds and one addition, the test functions and the mass matrix
// accumulate pairs.  Nodal values and table rows are pairs in memory too (odd NP
// padded with zeros), read in 64-bit loads.  The stress takes 2 d12 = E_12 + E_21,
// summed once at the nodes.
// Before (scalar, 122 registers at p = 2) -> after (107): 2,097,152 triangles,
// p = 2 250 -> 227 us; 524,288, p = 3 341 -> 252 us (128-thread blocks); 73,728,
// p = 2 14.5 -> 10.3 us.  What is left is latency: 23 % of the warps, half of the
// issue slots and half of the DRAM bandwidth in use.
#pragma once

namespace dgswe {

__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(d)
      : "l"(reinterpret_cast<unsigned long long&>(a)), "l"(reinterpret_cast<unsigned long long&>(b)),
        "l"(reinterpret_cast<unsigned long long&>(c)));
  return reinterpret_cast<float2&>(d);
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  unsigned long long d;
  asm("mul.rn.f32x2 %0, %1, %2;"
      : "=l"(d)
      : "l"(reinterpret_cast<unsigned long long&>(a)), "l"(reinterpret_cast<unsigned long long&>(b)));
  return reinterpret_cast<float2&>(d);
}
__device__ __forceinline__ float2 both(float x) { return make_float2(x, x); }
// component i of an array of pairs
template <int N>
__device__ __forceinline__ float& comp(float2 (&a)[N], int i) {
  return (i & 1) ? a[i / 2].y : a[i / 2].x;
}

// Operator tables of the pass: rows of pairs (see VolOps for their meaning), MP
// the products w_q l_a l_b (b <= a, row by row).
template <int DIM, int P>
struct VolF2 {
  using S = Sh<DIM, P>;
  static constexpr int NP = S::NP, NQ = S::NQ, NH = (NP + 1) / 2, NM = NP * (NP + 1) / 2, NMH = (NM + 1) / 2;
  float2 Vq[NQ * NH], Wr[NQ * NH], Ws[NQ * NH], Wm[NQ * NH], Drq[NQ * NH], Dsq[NQ * NH];
  float2 MP[NQ * NMH];
  float2 Minv[NP * NH];
  VolOps<DIM, P, float> o;  // the scalar tables (face lift, near-dry solve)
};

template <int NP>
__device__ __forceinline__ void load_pairs(const float* p, float2 (&out)[(NP + 1) / 2]) {
  if constexpr (NP % 2 == 0) {
    const float2* q = reinterpret_cast<const float2*>(p);
#pragma unroll
    for (int i = 0; i < NP / 2; ++i) out[i] = q[i];
  } else {
#pragma unroll
    for (int i = 0; i < NP / 2; ++i) out[i] = make_float2(p[2 * i], p[2 * i + 1]);
    out[NP / 2] = make_float2(p[NP - 1], 0.f);
  }
}
template <int NP>
__device__ __forceinline__ void load_pairs_cg(const float* p, float2 (&out)[(NP + 1) / 2]) {
#pragma unroll
  for (int i = 0; i < (NP + 1) / 2; ++i)
    out[i] = make_float2(__ldcg(p + 2 * i), 2 * i + 1 < NP ? __ldcg(p + 2 * i + 1) : 0.f);
}
template <int NP>
__device__ __forceinline__ void store_pairs(float* p, float2 (&v)[(NP + 1) / 2]) {
  if constexpr (NP % 2 == 0) {
    float2* q = reinterpret_cast<float2*>(p);
#pragma unroll
    for (int i = 0; i < NP / 2; ++i) q[i] = v[i];
  } else {
#pragma unroll
    for (int a = 0; a < NP; ++a) p[a] = comp(v, a);
  }
}
// sum_a row_a x_a.  Up to three nodes one after the other: as many instructions as in
// pairs, and one rounding less (rms error of dh/dt, 1D p = 1: 0.066 against 0.058
// units of 2^-24 of its terms).
template <int NP>
__device__ __forceinline__ float dot_pairs(const float2* row, const float2 (&x)[(NP + 1) / 2]) {
  [[maybe_unused]] constexpr int NH = (NP + 1) / 2;
  if constexpr (NP <= 3) {
    float s = fmaf(row[0].y, x[0].y, row[0].x * x[0].x);
    if constexpr (NP == 3) s = fmaf(row[1].x, x[1].x, s);
    return s;
  } else {
    float2 s = mul2(row[0], x[0]);
#pragma unroll
    for (int i = 1; i < NH; ++i) s = fma2(row[i], x[i], s);
    return s.x + s.y;
  }
}

// The element's nodal pairs: V, and the gradient components the stress needs
// (du/dx, or d11, d22, E_12 + E_21).
template <int DIM, int P, bool COH>
__device__ __forceinline__ void load_element_f32(const float* const (&Vp)[Sh<DIM, P>::NV],
                                                 const float* const (&Ep)[Sh<DIM, P>::NE],
                                                 float2 (&V2)[Sh<DIM, P>::NV][(Sh<DIM, P>::NP + 1) / 2],
                                                 float2 (&E2)[DIM == 1 ? 1 : 3][(Sh<DIM, P>::NP + 1) / 2]) {
  using S = Sh<DIM, P>;
  constexpr int NP = S::NP, NV = S::NV, NE = S::NE, NH = (NP + 1) / 2;
  auto get = [](const float* p, float2 (&out)[NH]) {
    if constexpr (COH) load_pairs_cg<NP>(p, out);
    else load_pairs<NP>(p, out);
  };
#pragma unroll
  for (int v = 0; v < NV; ++v) get(Vp[v], V2[v]);
  get(Ep[0], E2[0]);
  if constexpr (DIM == 2) {
    float2 x[NH];
    get(Ep[1], x);
    get(Ep[2], E2[2]);
    get(Ep[NE - 1], E2[1]);
#pragma unroll
    for (int i = 0; i < NH; ++i) E2[2][i] = make_float2(E2[2][i].x + x[i].x, E2[2][i].y + x[i].y);
  }
}

// Arguments and modes as volume_element_fx; V2, E2 as load_element_f32 gives them.
template <int DIM, int P, bool COH>
__device__ __forceinline__ void volume_element_f32(int e, int K, int F,
                                                   float2 (&V2)[Sh<DIM, P>::NV][(Sh<DIM, P>::NP + 1) / 2],
                                                   const float2 (&E2)[DIM == 1 ? 1 : 3][(Sh<DIM, P>::NP + 1) / 2],
                                                   const float* __restrict__ bed_e,
                                                   const float* const (&V0e)[Sh<DIM, P>::NV], float* out,
                                                   const float* __restrict__ geo, const int32_t* __restrict__ fid,
                                                   const float* __restrict__ wflux, const VolF2<DIM, P>& ops,
                                                   const Phys<float>& ph, int ins, int mode, float c0, float c1,
                                                   const DevScalars* __restrict__ sc) {
  using S = Sh<DIM, P>;
  using T = VolF2<DIM, P>;
  constexpr int NP = S::NP, NQ = S::NQ, NF = S::NF, NFP = S::NFP, NFQ = S::NFQ, NV = S::NV, NH = T::NH;
  constexpr int ND = DIM == 1 ? 1 : 3;
  const size_t KN = (size_t)K * NP;
  const size_t eo = (size_t)e * NP;
  float G[2][2];
  G[0][0] = geo[e];
  if constexpr (DIM == 2) {
    G[0][1] = geo[K + e];
    G[1][0] = geo[2 * K + e];
    G[1][1] = geo[3 * K + e];
  }
  float2 r[NV][NH];
#pragma unroll
  for (int v = 0; v < NV; ++v)
#pragma unroll
    for (int i = 0; i < NH; ++i) r[v][i] = both(0.f);
  const bool has_bed = bed_e != nullptr;
  float2 H2[NH];
#pragma unroll
  for (int i = 0; i < NH; ++i) H2[i] = both(0.f);
  if (has_bed) load_pairs<NP>(bed_e, H2);

  // ---- volume integrals: -<grad N, F - Q> - <N, S>  (Eq. WeakForm51)
#pragma unroll 1
  for (int q = 0; q < NQ; ++q) {
    const float2* lq = ops.Vq + q * NH;
    float Vq[NV], d[ND];
#pragma unroll
    for (int v = 0; v < NV; ++v) Vq[v] = dot_pairs<NP>(lq, V2[v]);
#pragma unroll
    for (int c = 0; c < ND; ++c) d[c] = dot_pairs<NP>(lq, E2[c]);
    float Hr = 0.f, Hs = 0.f;
    if (has_bed) {
      Hr = dot_pairs<NP>(ops.Drq + q * NH, H2);
      if constexpr (DIM == 2) Hs = dot_pairs<NP>(ops.Dsq + q * NH, H2);
    }
    const float h = Vq[0], hr = h * ph.rho_inv, p = 0.5f * ph.gc * h * h;
    float fr[NV], fs[NV], Sv[DIM];
    if constexpr (DIM == 1) {
      const float hu = h * Vq[1];
      fr[0] = -G[0][0] * hu;
      fr[1] = G[0][0] * (hr * stress_mu1<float>(d[0], ph) * 2.f * d[0] - hu * Vq[1] - p);
      Sv[0] = h * (ph.gc * G[0][0] * Hr + ph.gs);
    } else {
      constexpr int Y = 1 % ND, XY = 2 % ND, U2 = 2 % NV;
      const float tr = d[0] + d[Y], e12 = 0.5f * d[XY];
      const float s2 = 0.5f * (d[0] * d[0] + d[Y] * d[Y] + tr * tr + d[XY] * e12);
      const float m = hr * stress_mu2<float>(s2, ph);
      const float hu = h * Vq[1], hv = h * Vq[U2];
      const float T00 = m * (d[0] + tr) - hu * Vq[1] - p, T01 = m * e12 - hu * Vq[U2],
                  T11 = m * (d[Y] + tr) - hv * Vq[U2] - p;
      fr[0] = -(G[0][0] * hu + G[0][1] * hv);
      fs[0] = -(G[1][0] * hu + G[1][1] * hv);
      fr[1] = G[0][0] * T00 + G[0][1] * T01;
      fs[1] = G[1][0] * T00 + G[1][1] * T01;
      fr[U2] = G[0][0] * T01 + G[0][1] * T11;
      fs[U2] = G[1][0] * T01 + G[1][1] * T11;
      // minus the source
      Sv[0] = h * (ph.gc * (G[0][0] * Hr + G[1][0] * Hs) + ph.gs);
      Sv[1 % DIM] = h * (ph.gc * (G[0][1] * Hr + G[1][1] * Hs));
    }
#pragma unroll
    for (int i = 0; i < NH; ++i) {
      const float2 wr = ops.Wr[q * NH + i], ws = ops.Ws[q * NH + i], wm = ops.Wm[q * NH + i];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        float2 t = fma2(wr, both(fr[v]), r[v][i]);
        if constexpr (DIM == 2) t = fma2(ws, both(fs[v]), t);
        if (v > 0) t = fma2(wm, both(Sv[(v + DIM - 1) % DIM]), t);
        r[v][i] = t;
      }
    }
  }
  const float J = geo[4 * K + e];
  if constexpr (DIM == 2) {
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
      for (int i = 0; i < NH; ++i) r[v][i] = mul2(r[v][i], both(J));
  }

  // ---- face terms <N^-, F_bar.n - Q_bar.n> (weights and sJ folded into wflux)
  const size_t FQ = (size_t)F * NFQ;
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    const uint32_t raw = (uint32_t)fid[f * K + e];
    const bool own = (raw & 0x80000000u) == 0;
    const size_t base = (size_t)(raw & 0x7fffffffu) * NFQ;
    float fv[NV][NFQ];
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
      for (int m = 0; m < NFQ; ++m) {
        const float x = DG_LDC(COH, wflux, v * FQ + base + (own ? m : NFQ - 1 - m));
        fv[v][m] = own ? x : -x;
      }
#pragma unroll
    for (int k = 0; k < NFP; ++k) {
      const int a = face_node(DIM, P, f, k);
#pragma unroll
      for (int v = 0; v < NV; ++v)
#pragma unroll
        for (int m = 0; m < NFQ; ++m) {
          // 1D: one face value a node, added to J r in one rounding
          float& x = comp(r[v], a);
          if constexpr (DIM == 1) x = fmaf(x, J, ops.o.LfT[0] * fv[v][m]);
          else x += ops.o.LfT[k * NFQ + m] * fv[v][m];
        }
    }
  }
  if constexpr (DIM == 1) {
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
      for (int a = 1; a < NP - 1; ++a) comp(r[v], a) *= J;
  }

  // mode 2: the spatial residual r_V itself (physical scaling)
  if (mode == 2) {
#pragma unroll
    for (int v = 0; v < NV; ++v) store_pairs<NP>(out + v * KN + eo, r[v]);
    return;
  }

  // ---- mass solve: M dh/dt = -r_h ; M_h du/dt = -r_u - M_u dh/dt
  const float Jinv = geo[6 * K + e];
  float2 dV[NV][NH];
  float hmin = V2[0][0].x;
#pragma unroll
  for (int a = 1; a < NP; ++a) hmin = fminf(hmin, comp(V2[0], a));
  if (hmin < ph.h_dry) {
    // near-dry element: FP64 (mass_solve_dry)
    float Vn[NV][NP], rn[NV][NP], dn[NV][NP];
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
      for (int a = 0; a < NP; ++a) {
        Vn[v][a] = comp(V2[v], a);
        rn[v][a] = comp(r[v], a);
      }
    mass_solve_dry<DIM, P>(Vn, rn, ops.o, ph.h_floor, Jinv, dn);
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
      for (int a = 0; a < NP; ++a) comp(dV[v], a) = dn[v][a];
  } else {
    if constexpr (NP % 2 == 1) dV[0][NH - 1].y = 0.f;
#pragma unroll
    for (int a = 0; a < NP; ++a) comp(dV[0], a) = -Jinv * dot_pairs<NP>(ops.Minv + a * NH, r[0]);
    float2 M[T::NMH], rhs[DIM][NH];
#pragma unroll
    for (int i = 0; i < T::NMH; ++i) M[i] = both(0.f);
#pragma unroll
    for (int j = 0; j < DIM; ++j)
#pragma unroll
      for (int i = 0; i < NH; ++i) rhs[j][i] = mul2(r[1 + j][i], both(-Jinv));
#pragma unroll 1
    for (int q = 0; q < NQ; ++q) {
      const float2* lq = ops.Vq + q * NH;
      const float hf = fmaxf(dot_pairs<NP>(lq, V2[0]), ph.h_floor), hd = -dot_pairs<NP>(lq, dV[0]);
#pragma unroll
      for (int i = 0; i < T::NMH; ++i) M[i] = fma2(ops.MP[q * T::NMH + i], both(hf), M[i]);
#pragma unroll
      for (int j = 0; j < DIM; ++j) {
        const float2 z = both(hd * dot_pairs<NP>(lq, V2[1 + j]));
#pragma unroll
        for (int i = 0; i < NH; ++i) rhs[j][i] = fma2(ops.Wm[q * NH + i], z, rhs[j][i]);
      }
    }
    // Cholesky of the reference-scaled M_h (lower triangle, row by row), the
    // diagonal kept as reciprocals
    float dinv[NP];
#pragma unroll
    for (int a = 0; a < NP; ++a) {
#pragma unroll
      for (int b = 0; b < a; ++b) {
        float s = comp(M, a * (a + 1) / 2 + b);
#pragma unroll
        for (int c = 0; c < b; ++c) s -= comp(M, a * (a + 1) / 2 + c) * comp(M, b * (b + 1) / 2 + c);
        comp(M, a * (a + 1) / 2 + b) = s * dinv[b];
      }
      float s = comp(M, a * (a + 1) / 2 + a);
#pragma unroll
      for (int c = 0; c < a; ++c) s -= comp(M, a * (a + 1) / 2 + c) * comp(M, a * (a + 1) / 2 + c);
      dinv[a] = rsqrtf(s);
    }
#pragma unroll
    for (int j = 0; j < DIM; ++j) {
      float y[NP];
#pragma unroll
      for (int a = 0; a < NP; ++a) {
        float s = comp(rhs[j], a);
#pragma unroll
        for (int c = 0; c < a; ++c) s -= comp(M, a * (a + 1) / 2 + c) * y[c];
        y[a] = s * dinv[a];
      }
#pragma unroll
      for (int a = NP - 1; a >= 0; --a) {
        float s = y[a];
#pragma unroll
        for (int c = a + 1; c < NP; ++c) s -= comp(M, c * (c + 1) / 2 + a) * comp(dV[1 + j], c);
        comp(dV[1 + j], a) = s * dinv[a];
      }
    }
  }

  // ---- output
  if (mode == 1) {
    const float dt = (float)DG_LDC(COH, &sc[ins].dt, 0);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      float2 v0[NH];
      if (c0 != 0.f) {
        if constexpr (COH) load_pairs_cg<NP>(V0e[v], v0);
        else load_pairs<NP>(V0e[v], v0);
      }
#pragma unroll
      for (int i = 0; i < NH; ++i) {
        float2 y = mul2(both(c1), fma2(both(dt), dV[v][i], V2[v][i]));
        if (c0 != 0.f) y = fma2(both(c0), v0[i], y);
        dV[v][i] = y;
      }
    }
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) store_pairs<NP>(out + v * KN + eo, dV[v]);
}

// ------------------------------------------------------------------ host: tables

template <int DIM, int P>
void fill_vol_f2(const RefOps& ro, const VolOps<DIM, P, float>& o, VolF2<DIM, P>& t) {
  using T = VolF2<DIM, P>;
  constexpr int NP = T::NP, NQ = T::NQ, NH = T::NH;
  t.o = o;
  auto put = [](float2& p, int i, double v) { (i & 1 ? p.y : p.x) = (float)v; };
  for (int q = 0; q < NQ; ++q) {
    const double w = ro.wq[q];
    for (int a = 0, i = 0; a < NP; ++a) {
      const int j = q * NP + a, k = q * NH + a / 2;
      const double ds = DIM == 2 ? ro.Dsq[j] : 0.0;
      put(t.Vq[k], a, ro.Vq[j]);
      put(t.Wr[k], a, w * ro.Drq[j]);
      put(t.Ws[k], a, w * ds);
      put(t.Wm[k], a, w * ro.Vq[j]);
      put(t.Drq[k], a, ro.Drq[j]);
      put(t.Dsq[k], a, ds);
      for (int b = 0; b <= a; ++b, ++i) put(t.MP[q * T::NMH + i / 2], i, w * ro.Vq[j] * ro.Vq[q * NP + b]);
    }
  }
  for (int a = 0; a < NP; ++a)
    for (int b = 0; b < NP; ++b) put(t.Minv[a * NH + b / 2], b, ro.Minv[a * NP + b]);
}

}  // namespace dgswe
