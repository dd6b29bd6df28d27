// The FP64 volume pass of one element with its contractions in block fixed
// point (dg_fixed.cuh).  Included by dg_kernels.cuh.
//
// What stays in floating point is the pointwise stress and flux (about 38
// operations a volume point in 2D), the Cholesky solve and the stage update:
// 500 FP64 instructions per element at p = 2 (counted) where the pass in
// floating point took 2065 and kept the FP64 pipe 91 % busy; the contractions
// (interpolation, metric transform, test functions, face lift, mass matrices)
// are 1140 integer multiply-adds of three IMAD.WIDE each.  524,288 triangles,
// p = 2: 1969 -> 844 us, p = 1 691 -> 403 us (with the wet/dry stage kernel);
// 73,728 triangles, p = 2: 314 -> 160 us; 8,192: 84 -> 47 us.  The FP64 pipe is
// 50 % busy then: few warps (168 to 240 registers a thread) wait for one
// another's chains.
//
//   pass 1  per volume point: interpolate V and the symmetric gradient, form
//           the flux tensor, the source and h for M_h; keep them (local memory)
//           with the largest exponent of each component
//   pass 2  per volume point: metric transform J G (Q - F), test functions;
//           the face fluxes are lifted into the same accumulators
//   solve   M dh/dt = -r_h straight from the integer residual, then M_h and
//           M_u dh/dt per volume point, Cholesky in floating point
//
// Every component of the residual has a unit of its own, set by the largest of its
// terms, and the metric terms of each direction have theirs: on stretched elements,
// or with a momentum component far below the other, a unit for all would take bits
// from the small ones.
#pragma once

namespace dgswe {

// Constant tables of the pass.  Vq: interpolation; Wr, Ws, Wm: w_q dl_a/dr,
// w_q dl_a/ds, w_q l_a, and LfT the face lift, one scale cs_w; MP: w_q l_a l_b
// (b <= a, row by row).
template <int DIM, int P>
struct VolFx {
  using S = Sh<DIM, P>;
  static constexpr int NP = S::NP, NQ = S::NQ, NM = NP * (NP + 1) / 2;
  Fx Vq[NQ * NP], Wr[NQ * NP], Ws[NQ * NP], Wm[NQ * NP];
  Fx MP[NQ * NM];
  Fx Minv[NP * NP];
  Fx LfT[S::NFP * S::NFQ];
  int cs_v, cs_w, cs_m, cs_i;
};

// Shared-memory copy of the per-point rows: per volume point Vq, Wr, Ws, Wm and
// MP, each padded to 16 bytes, read in 128-bit loads (uniform in a warp).  1D
// reads the kernel parameters (the fill costs more than it saves there), and so
// does the staged kernel, whose shared memory holds its tiles (tab = nullptr).
template <int DIM, int P>
struct FxTab {
  using T = VolFx<DIM, P>;
  static constexpr bool USED = DIM == 2;
  static constexpr int PAD = (T::NP + 1) / 2 * 2, MPAD = (T::NM + 1) / 2 * 2;
  static constexpr int ROW = 4 * PAD + MPAD;
  static constexpr int SIZE = USED ? T::NQ * ROW : 2;
};
template <int DIM, int P>
__device__ __forceinline__ void fxtab_fill(Fx* tab, const VolFx<DIM, P>& ops) {
  using T = FxTab<DIM, P>;
  using O = VolFx<DIM, P>;
  if constexpr (T::USED) {
    for (int i = threadIdx.x; i < T::SIZE; i += blockDim.x) {
      const int q = i / T::ROW, c = i % T::ROW, k = c < 4 * T::PAD ? c / T::PAD : 4;
      const int a = c - k * T::PAD;
      Fx v{0, 0};
      if (k < 4 && a < O::NP) v = (k == 0 ? ops.Vq : k == 1 ? ops.Wr : k == 2 ? ops.Ws : ops.Wm)[q * O::NP + a];
      if (k == 4 && a < O::NM) v = ops.MP[q * O::NM + a];
      tab[i] = v;
    }
  }
}
// Row K of volume point q (K = 0..3: Vq, Wr, Ws, Wm; 4: MP).
template <int DIM, int P, int K, int N>
__device__ __forceinline__ void fx_row(const VolFx<DIM, P>& ops, const Fx* tab, int q, Fx (&out)[N]) {
  using T = FxTab<DIM, P>;
  if (T::USED && tab) {
    const int4* p = reinterpret_cast<const int4*>(tab + q * T::ROW + K * T::PAD);
#pragma unroll
    for (int c = 0; c < (N + 1) / 2; ++c) {
      const int4 v = p[c];
      out[2 * c] = Fx{v.x, v.y};
      if (2 * c + 1 < N) out[2 * c + 1] = Fx{v.z, v.w};
    }
    return;
  }
  const Fx* src = K == 0 ? ops.Vq : K == 1 ? ops.Wr : K == 2 ? ops.Ws : K == 3 ? ops.Wm : ops.MP;
#pragma unroll
  for (int a = 0; a < N; ++a) out[a] = src[q * N + a];
}

// Sums and maxima over the T neighbouring lanes that share an element.
// (the sum's two parts apart, so that it is exactly that of T = 1)
template <int T>
__device__ __forceinline__ long long lanes_sum(FxAcc v) {
  if constexpr (T > 1) {
    fx_fold(v);
    int low = (int)v.b;
#pragma unroll
    for (int o = 1; o < T; o *= 2) {
      v.a += __shfl_xor_sync(0xffffffffu, v.a, o);
      low += __shfl_xor_sync(0xffffffffu, low, o);
    }
    v.b = low;
  }
  return fx_sum(v);
}
// (N exponents, two in a word)
template <int T, int N>
__device__ __forceinline__ void lanes_max(int (&v)[N]) {
  if constexpr (T > 1) {
#pragma unroll
    for (int i = 0; i < N; i += 2) {
      unsigned w = (unsigned)v[i] | (i + 1 < N ? (unsigned)v[i + 1] << 16 : 0u);
#pragma unroll
      for (int o = 1; o < T; o *= 2) w = __vmaxu2(w, __shfl_xor_sync(0xffffffffu, w, o));
      v[i] = (int)(w & 0xffffu);
      if (i + 1 < N) v[i + 1] = (int)(w >> 16);
    }
  }
}
template <int N>
__device__ __forceinline__ int largest(const int (&v)[N]) {
  int m = v[0];
#pragma unroll
  for (int i = 1; i < N; ++i) m = max(m, v[i]);
  return m;
}

// Arguments and modes as volume_any (dg_kernels.cuh).  T = 1: one thread per
// element.  T = 2, 4: T neighbouring lanes share one (tl: the thread's place
// among them; all lanes of a warp come here, live = false for those past the
// last element): each takes every T-th volume point and face, the integer sums
// are added across the lanes (exactly, so the results are those of T = 1), and
// each writes every T-th node.
template <int DIM, int P, bool COH, int T = 1>
__device__ __forceinline__ void volume_element_fx(int e, int K, int F,
                                                  const double (&Vn)[Sh<DIM, P>::NV][Sh<DIM, P>::NP],
                                                  const double (&En)[Sh<DIM, P>::NE][Sh<DIM, P>::NP],
                                                  const double* __restrict__ src,
                                                  const double* const (&V0e)[Sh<DIM, P>::NV], double* out,
                                                  const double* __restrict__ geo, const int32_t* __restrict__ fid,
                                                  const double* __restrict__ wflux, const VolFx<DIM, P>& ops,
                                                  const Phys<double>& ph, int ins, int mode, double c0, double c1,
                                                  const DevScalars* __restrict__ sc, const Fx* tab, int tl = 0,
                                                  bool live = true) {
  using S = Sh<DIM, P>;
  constexpr int NP = S::NP, NQ = S::NQ, NF = S::NF, NFP = S::NFP, NFQ = S::NFQ, NV = S::NV;
  constexpr int NS = (NQ + T - 1) / T;  // volume points of a thread
  constexpr int NM = VolFx<DIM, P>::NM;
  constexpr int ND = DIM == 1 ? 1 : 3;  // gradient components the stress needs
  constexpr int NT = DIM == 1 ? 1 : 3;  // momentum flux tensor (symmetric)
  const size_t KN = (size_t)K * NP;
  const size_t eo = (size_t)e * NP;

  double hu_s[NS][DIM], T_s[NS][NT], S_s[NS][DIM], u_s[NS][DIM];
  double hm_s[NS];
  // largest exponents of each component of the flux (h u, then the tensor) and of the source
  int eX[DIM + NT], eS[DIM];
#pragma unroll
  for (int c = 0; c < DIM + NT; ++c) eX[c] = 0;
#pragma unroll
  for (int j = 0; j < DIM; ++j) eS[j] = 0;
  // largest exponent of max(h, h_floor): of the points themselves, for where the depth
  // is below the floor the nodal values can be far above what M_h holds
  int eM[1] = {0};
  bool finite = true;

  {  // ---- pass 1
    Fx vx[NV][NP], dx[ND][NP];
    FxScale sv[NV], sd[ND];
    // results in units of 2^(E - 1080) 2^-cs_v 2^56
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      int ev = 0;
#pragma unroll
      for (int a = 0; a < NP; ++a) ev = max(ev, fx_exp(Vn[v][a]));
#pragma unroll
      for (int a = 0; a < NP; ++a) vx[v][a] = fx_from<5>(Vn[v][a], ev);
      sv[v] = fx_scale(ev - 1024 - ops.cs_v, ev <= kFxMaxExp);
      finite = finite && ev <= kFxMaxExp;
    }
    if constexpr (DIM == 1) {
      int ed = 0;
#pragma unroll
      for (int a = 0; a < NP; ++a) ed = max(ed, fx_exp(En[0][a]));
#pragma unroll
      for (int a = 0; a < NP; ++a) dx[0][a] = fx_from<5>(En[0][a], ed);
      sd[0] = fx_scale(ed - 1024 - ops.cs_v, ed <= kFxMaxExp);
    } else {
      // d11, d22 and d12 = (E_12 + E_21) / 2, summed at the nodes
      constexpr int NE = S::NE;
      int e0 = 0, e3 = 0, e12 = 0;
#pragma unroll
      for (int a = 0; a < NP; ++a) {
        e0 = max(e0, fx_exp(En[0][a]));
        e3 = max(e3, fx_exp(En[NE - 1][a]));
        e12 = max(e12, max(fx_exp(En[1 % NE][a]), fx_exp(En[2 % NE][a])));
      }
#pragma unroll
      for (int a = 0; a < NP; ++a) {
        dx[0][a] = fx_from<5>(En[0][a], e0);
        dx[1 % ND][a] = fx_from<5>(En[NE - 1][a], e3);
        const Fx x = fx_from<4>(En[1 % NE][a], e12), y = fx_from<4>(En[2 % NE][a], e12);
        dx[2 % ND][a] = Fx{x.h + y.h, x.l + y.l};
      }
      sd[0] = fx_scale(e0 - 1024 - ops.cs_v, e0 <= kFxMaxExp);
      sd[1 % ND] = fx_scale(e3 - 1024 - ops.cs_v, e3 <= kFxMaxExp);
      sd[2 % ND] = fx_scale(e12 - 1024 - ops.cs_v, e12 <= kFxMaxExp);
    }
#pragma unroll 1
    for (int q = tl, i = 0; q < NQ; q += T, ++i) {
      Fx row[NP];
      fx_row<DIM, P, 0>(ops, tab, q, row);
      double Vq[NV], d[ND];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        FxAcc s{0, 0};
#pragma unroll
        for (int a = 0; a < NP; ++a) fx_mac(s, vx[v][a], row[a]);
        Vq[v] = fx_to(fx_sum(s), sv[v]);
      }
#pragma unroll
      for (int c = 0; c < ND; ++c) {
        FxAcc s{0, 0};
#pragma unroll
        for (int a = 0; a < NP; ++a) fx_mac(s, dx[c][a], row[a]);
        d[c] = fx_to(fx_sum(s), sd[c]);
      }
      const double h = Vq[0];
      // max(h, h_floor) as integers: h_floor > 0, so a negative h orders below it
      const double hm = __longlong_as_double(max(__double_as_longlong(h), __double_as_longlong(ph.h_floor)));
      hm_s[i] = hm;
      eM[0] = max(eM[0], fx_exp(hm));
      double hu[DIM], Tq[NT], Sv[DIM];
#pragma unroll
      for (int j = 0; j < DIM; ++j) hu[j] = -h * Vq[1 + j];
      const double p = (0.5 * ph.gc * h) * h;
      if constexpr (DIM == 1) {
        Tq[0] = h * ph.rho_inv * stress_mu1<double>(d[0], ph) * (2.0 * d[0]) + (hu[0] * Vq[1] - p);
      } else {
        constexpr int Y = 1 % ND, XY = 2 % ND, U2 = 2 % NV;
        // a_i = d_ii + tr D; d11 a_1 + d22 a_2 = d11^2 + d22^2 + tr^2; s2 = ||D||_c^2 / 2
        const double a1 = fma(2.0, d[0], d[Y]), a2 = fma(2.0, d[Y], d[0]);
        const double s2 = fma(0.5, fma(d[0], a1, d[Y] * a2), d[XY] * d[XY]);
        const double m = h * ph.rho_inv * stress_mu2<double>(s2, ph);
        Tq[0] = fma(m, a1, fma(hu[0], Vq[1], -p));
        Tq[1 % NT] = fma(m, d[XY], hu[0] * Vq[U2]);
        Tq[2 % NT] = fma(m, a2, fma(hu[1 % DIM], Vq[U2], -p));
      }
#pragma unroll
      for (int j = 0; j < DIM; ++j) {
        if (src) Sv[j] = h * src[(size_t)(j * NQ + q) * K + e];
        else Sv[j] = j == 0 ? -ph.gs * h : 0.0;
        hu_s[i][j] = hu[j];
        S_s[i][j] = Sv[j];
        u_s[i][j] = Vq[1 + j];
        eX[j] = max(eX[j], fx_exp(hu[j]));
        eS[j] = max(eS[j], fx_exp(Sv[j]));
      }
#pragma unroll
      for (int c = 0; c < NT; ++c) {
        T_s[i][c] = Tq[c];
        eX[DIM + c] = max(eX[DIM + c], fx_exp(Tq[c]));
      }
    }
  }
  lanes_max<T>(eX);
  lanes_max<T>(eS);
  lanes_max<T>(eM);

  // ---- pass 2: J times (metric transform, test functions, face lift)
  FxAcc r[NV][NP];
#pragma unroll
  for (int v = 0; v < NV; ++v)
#pragma unroll
    for (int a = 0; a < NP; ++a) r[v][a] = FxAcc{0, 0};
  const double J = geo[4 * K + e];
  double JG[DIM][DIM];
#pragma unroll
  for (int k = 0; k < DIM; ++k)
#pragma unroll
    for (int i = 0; i < DIM; ++i) JG[k][i] = J * geo[(2 * k + i) * K + e];
  int eG[DIM];  // of each direction i
#pragma unroll
  for (int i = 0; i < DIM; ++i) {
    eG[i] = 0;
#pragma unroll
    for (int k = 0; k < DIM; ++k) eG[i] = max(eG[i], fx_exp(JG[k][i]));
  }
  const int eJ = fx_exp(J);
  // weighted face fluxes, in the owner's orientation
  double fv[NF][NV][NFQ];
  int eW[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) eW[v] = 0;
  const size_t FQ = (size_t)F * NFQ;
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    if (T > 1 && f % T != tl) continue;
    const uint32_t raw = (uint32_t)fid[f * K + e];
    const bool own = (raw & 0x80000000u) == 0;
    const size_t base = (size_t)(raw & 0x7fffffffu) * NFQ;
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
      for (int m = 0; m < NFQ; ++m) {
        const double x = DG_LDC(COH, wflux, v * FQ + base + (own ? m : NFQ - 1 - m));
        fv[f][v][m] = __hiloint2double(__double2hiint(x) ^ (own ? 0 : (int)0x80000000u), __double2loint(x));
        eW[v] = max(eW[v], fx_exp(x));
      }
  }
  lanes_max<T>(eW);
  // a unit for each row (depth, momentum components): its terms below 2^(tot - 2043)
  // in units of 2^(tot - 2101).  flux_of: component of the flux in row v, direction i.
  auto flux_of = [](int v, int i) { return v == 0 ? i : DIM + (v - 1 + i) % (NT + 1); };
  int tot[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    tot[v] = eW[v] + 1021;
#pragma unroll
    for (int i = 0; i < DIM; ++i) tot[v] = max(tot[v], eX[flux_of(v, i)] + eG[i]);
    if (v > 0) tot[v] = max(tot[v], eS[(v + DIM - 1) % DIM] + eJ);
  }
  finite = finite && max(max(largest(eX), largest(eS)), largest(eW)) <= kFxMaxExp;
#pragma unroll
  for (int f = 0; f < NF; ++f)
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
      for (int m = 0; m < NFQ; ++m) {
        if (T > 1 && f % T != tl) continue;
        const Fx x = fx_from<5>(fv[f][v][m], tot[v] - 1021);
#pragma unroll
        for (int k = 0; k < NFP; ++k) fx_mac(r[v][face_node(DIM, P, f, k)], x, ops.LfT[k * NFQ + m]);
      }
  {
    Fx JGx[DIM][DIM];
#pragma unroll
    for (int k = 0; k < DIM; ++k)
#pragma unroll
      for (int i = 0; i < DIM; ++i) JGx[k][i] = fx_from<5>(JG[k][i], eG[i]);
    const Fx Jx = fx_from<5>(-J, eJ);
    // at most 2 NFQ + 5 (DIM + 1) terms before the first fold, 5 (DIM + 1) after it
    static_assert(2 * S::NFQ <= 15, "the lift terms need a fold of their own");
#pragma unroll 1
    for (int q = tl, k = 0; q < NQ; q += T, ++k) {
      if (DIM == 2 && k % 5 == 0) {
#pragma unroll
        for (int v = 0; v < NV; ++v)
#pragma unroll
          for (int a = 0; a < NP; ++a) fx_fold(r[v][a]);
      }
      Fx wr[NP], ws[NP], wm[NP];
      fx_row<DIM, P, 1>(ops, tab, q, wr);
      if constexpr (DIM == 2) fx_row<DIM, P, 2>(ops, tab, q, ws);
      fx_row<DIM, P, 3>(ops, tab, q, wm);
      // rows: depth, then momentum
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        Fx x[DIM];
#pragma unroll
        for (int i = 0; i < DIM; ++i)
          x[i] = fx_from<5>(v == 0 ? hu_s[k][i] : T_s[k][(v - 1 + i) % (NT + 1)], tot[v] - eG[i]);
        FxAcc fr{0, 0}, fs{0, 0};
#pragma unroll
        for (int i = 0; i < DIM; ++i) {
          fx_mac(fr, x[i], JGx[0][i]);
          if constexpr (DIM == 2) fx_mac(fs, x[i], JGx[DIM - 1][i]);
        }
        const Fx frx = fx_operand<61>(fx_sum(fr));
        Fx fsx{0, 0}, sx{0, 0};
        if constexpr (DIM == 2) fsx = fx_operand<61>(fx_sum(fs));
        if (v > 0) {
          FxAcc s{0, 0};
          fx_mac(s, fx_from<5>(S_s[k][(v + DIM - 1) % DIM], tot[v] - eJ), Jx);
          sx = fx_operand<61>(fx_sum(s));
        }
#pragma unroll
        for (int a = 0; a < NP; ++a) {
          fx_mac(r[v][a], frx, wr[a]);
          if constexpr (DIM == 2) fx_mac(r[v][a], fsx, ws[a]);
          if (v > 0) fx_mac(r[v][a], sx, wm[a]);
        }
      }
    }
  }
  long long rs[NV][NP];
#pragma unroll
  for (int v = 0; v < NV; ++v)
#pragma unroll
    for (int a = 0; a < NP; ++a) rs[v][a] = lanes_sum<T>(r[v][a]);
  FxScale sr[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) sr[v] = fx_scale(tot[v] - 2045 - ops.cs_w, finite);

  // mode 2: the spatial residual r_V itself (physical scaling), for the
  // implicit integrators that assemble their own time term
  if (mode == 2) {
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
      for (int a = 0; a < NP; ++a)
        if (live && (T == 1 || a % T == tl)) out[v * KN + eo + a] = fx_to(rs[v][a], sr[v]);
    return;
  }

  // ---- mass solve, J dV/dt: x_h = -Minv r_h ; M_h x_u = -r_u - <psi, x_h u>
  double x[NV][NP], ru[DIM][NP];
  Fx dh[NP];
  int kh = tot[0] - 2045 - ops.cs_w;  // binary orders of what dh holds
  {
    // r_h brought up to full length (the fluxes mostly cancel in it)
    long long rh[NP];
    unsigned long long m = 0;
#pragma unroll
    for (int a = 0; a < NP; ++a) {
      rh[a] = rs[0][a];
      m |= fx_mag(rh[a]);
#pragma unroll
      for (int j = 0; j < DIM; ++j) ru[j][a] = fx_to(rs[1 + j][a], sr[1 + j]);
    }
    int n = fx_norm(m);
    Fx rx[NP];
#pragma unroll
    for (int a = 0; a < NP; ++a) rx[a] = fx_operand<62>(rh[a] << n);
    // Minv r_h in units of (unit of r_h) 2^-n 2^4 2^-cs_i 2^56
    kh += 60 - n - ops.cs_i;
    const FxScale si = fx_scale(kh, finite);
    m = 0;
#pragma unroll
    for (int a = 0; a < NP; ++a) {
      FxAcc s{0, 0};
#pragma unroll
      for (int b = 0; b < NP; ++b) fx_mac(s, rx[b], ops.Minv[a * NP + b]);
      rh[a] = fx_sum(s);
      m |= fx_mag(rh[a]);
      x[0][a] = -fx_to(rh[a], si);
    }
    n = fx_norm(m);
#pragma unroll
    for (int a = 0; a < NP; ++a) dh[a] = fx_operand<62>(rh[a] << n);
    kh += 60 - n - ops.cs_v;
  }
  const FxScale sq = fx_scale(kh, finite);
  int eZ[DIM];
#pragma unroll
  for (int j = 0; j < DIM; ++j) eZ[j] = 0;
#pragma unroll 1
  for (int q = tl, k = 0; q < NQ; q += T, ++k) {
    Fx row[NP];
    fx_row<DIM, P, 0>(ops, tab, q, row);
    FxAcc s{0, 0};
#pragma unroll
    for (int a = 0; a < NP; ++a) fx_mac(s, dh[a], row[a]);
    const double dq = fx_to(fx_sum(s), sq);
#pragma unroll
    for (int j = 0; j < DIM; ++j) {
      const double z = dq * u_s[k][j];
      u_s[k][j] = z;
      eZ[j] = max(eZ[j], fx_exp(z));
    }
  }
  lanes_max<T>(eZ);
  const FxScale sm = fx_scale(eM[0] - 1024 - ops.cs_m, finite);
  // -r_u - <psi, x_h u>, and after it M_h (one after the other: their
  // accumulators together would take 132 registers at p = 2)
  {
    FxAcc za[DIM][NP];
#pragma unroll
    for (int j = 0; j < DIM; ++j)
#pragma unroll
      for (int a = 0; a < NP; ++a) za[j][a] = FxAcc{0, 0};
#pragma unroll 1
    for (int q = tl, k = 0; q < NQ; q += T, ++k) {
      Fx wm[NP];
      fx_row<DIM, P, 3>(ops, tab, q, wm);
      if (NS > 15 && k % 12 == 0) {
#pragma unroll
        for (int j = 0; j < DIM; ++j)
#pragma unroll
          for (int a = 0; a < NP; ++a) fx_fold(za[j][a]);
      }
#pragma unroll
      for (int j = 0; j < DIM; ++j) {
        const Fx z = fx_from<5>(u_s[k][j], eZ[j]);
#pragma unroll
        for (int a = 0; a < NP; ++a) fx_mac(za[j][a], z, wm[a]);
      }
    }
#pragma unroll
    for (int j = 0; j < DIM; ++j) {
      const FxScale sz = fx_scale(eZ[j] - 1024 - ops.cs_w, finite && eZ[j] <= kFxMaxExp);
#pragma unroll
      for (int a = 0; a < NP; ++a) ru[j][a] = fx_to(lanes_sum<T>(za[j][a]), sz) - ru[j][a];
    }
  }
  FxAcc Ma[NM];
#pragma unroll
  for (int i = 0; i < NM; ++i) Ma[i] = FxAcc{0, 0};
#pragma unroll 1
  for (int q = tl, k = 0; q < NQ; q += T, ++k) {
    Fx mp[NM];
    fx_row<DIM, P, 4>(ops, tab, q, mp);
    const Fx hm = fx_from<5>(hm_s[k], eM[0]);
    if (NS > 15 && k % 12 == 0) {
#pragma unroll
      for (int i = 0; i < NM; ++i) fx_fold(Ma[i]);
    }
#pragma unroll
    for (int i = 0; i < NM; ++i) fx_mac(Ma[i], hm, mp[i]);
  }
  // Cholesky of the reference-scaled M_h (lower triangle); the diagonal is
  // kept as reciprocals so the factorization and both triangular solves
  // multiply instead of divide
  double Mh[NP][NP], dinv[NP];
#pragma unroll
  for (int a = 0, i = 0; a < NP; ++a) {
#pragma unroll
    for (int b = 0; b <= a; ++b, ++i) Mh[a][b] = fx_to(lanes_sum<T>(Ma[i]), sm);
#pragma unroll
    for (int b = 0; b < a; ++b) {
      double s = Mh[a][b];
#pragma unroll
      for (int c = 0; c < b; ++c) s -= Mh[a][c] * Mh[b][c];
      Mh[a][b] = s * dinv[b];
    }
    double d = Mh[a][a];
#pragma unroll
    for (int c = 0; c < a; ++c) d -= Mh[a][c] * Mh[a][c];
    dinv[a] = dg_rsqrt<double>(d);
  }
#pragma unroll
  for (int j = 0; j < DIM; ++j) {
    double y[NP];
#pragma unroll
    for (int a = 0; a < NP; ++a) {
      double s = ru[j][a];
#pragma unroll
      for (int c = 0; c < a; ++c) s -= Mh[a][c] * y[c];
      y[a] = s * dinv[a];
    }
#pragma unroll
    for (int a = NP - 1; a >= 0; --a) {
      double s = y[a];
#pragma unroll
      for (int c = a + 1; c < NP; ++c) s -= Mh[c][a] * x[1 + j][c];
      x[1 + j][a] = s * dinv[a];
    }
  }

  // ---- output: dV/dt = x / J
  const double Jinv = geo[6 * K + e];
  if (mode == 0) {
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
      for (int a = 0; a < NP; ++a)
        if (live && (T == 1 || a % T == tl)) out[v * KN + eo + a] = Jinv * x[v][a];
    return;
  }
  const double cx = DG_LDC(COH, &sc[ins].dt, 0) * Jinv;
#pragma unroll
  for (int v = 0; v < NV; ++v)
#pragma unroll
    for (int a = 0; a < NP; ++a) {
      if (T > 1 && a % T != tl) continue;
      double y = c1 * (Vn[v][a] + cx * x[v][a]);
      if (c0 != 0.0) y += c0 * DG_LDC(COH, V0e[v], a);
      x[v][a] = y;
    }
#pragma unroll
  for (int v = 0; v < NV; ++v)
#pragma unroll
    for (int a = 0; a < NP; ++a)
      if (live && (T == 1 || a % T == tl)) out[v * KN + eo + a] = x[v][a];
}

// ------------------------------------------------------------------ host: tables

template <int DIM, int P>
void fill_vol_fx(const RefOps& o, VolFx<DIM, P>& t) {
  using S = Sh<DIM, P>;
  constexpr int NP = S::NP, NQ = S::NQ, NM = VolFx<DIM, P>::NM;
  double vmax = 0, vrow = 0, wmax = 0, wrow = 0, mmax = 0, mrow = 0, imax = 0, irow = 0;
  std::vector<double> mp((size_t)NQ * NM), msum(NM, 0.0), wsum(NP, 0.0), lsum(NP, 0.0);
  for (int q = 0; q < NQ; ++q) {
    double r = 0;
    for (int a = 0, i = 0; a < NP; ++a) {
      const double l = o.Vq[q * NP + a], w = o.wq[q];
      const double dr = w * o.Drq[q * NP + a], ds = DIM == 2 ? w * o.Dsq[q * NP + a] : 0.0;
      vmax = std::max(vmax, std::fabs(l));
      r += std::fabs(l);
      wmax = std::max({wmax, std::fabs(dr), std::fabs(ds), std::fabs(w * l)});
      wsum[a] += std::fabs(dr) + std::fabs(ds) + std::fabs(w * l);
      for (int b = 0; b <= a; ++b, ++i) {
        mp[(size_t)q * NM + i] = w * l * o.Vq[q * NP + b];
        mmax = std::max(mmax, std::fabs(mp[(size_t)q * NM + i]));
        msum[i] += std::fabs(mp[(size_t)q * NM + i]);
      }
    }
    vrow = std::max(vrow, r);
  }
  for (int f = 0; f < S::NF; ++f)
    for (int k = 0; k < S::NFP; ++k)
      for (int m = 0; m < S::NFQ; ++m) {
        wmax = std::max(wmax, std::fabs(o.Lf[m * S::NFP + k]));
        lsum[o.fmask[f * S::NFP + k]] += std::fabs(o.Lf[m * S::NFP + k]);
      }
  for (int a = 0; a < NP; ++a) {
    wrow = std::max(wrow, wsum[a] + lsum[a]);
    double r = 0;
    for (int b = 0; b < NP; ++b) {
      imax = std::max(imax, std::fabs(o.Minv[a * NP + b]));
      r += std::fabs(o.Minv[a * NP + b]);
    }
    irow = std::max(irow, r);
  }
  for (int i = 0; i < NM; ++i) mrow = std::max(mrow, msum[i]);
  t.cs_v = fx_table_scale(vmax, vrow, 58);
  t.cs_w = fx_table_scale(wmax, wrow, 58);
  t.cs_m = fx_table_scale(mmax, mrow, 58);
  t.cs_i = fx_table_scale(imax, irow, 58);
  for (int i = 0; i < NQ * NP; ++i) {
    const double w = o.wq[i / NP];
    t.Vq[i] = fx_const(o.Vq[i], t.cs_v);
    t.Wr[i] = fx_const(w * o.Drq[i], t.cs_w);
    t.Ws[i] = fx_const(DIM == 2 ? w * o.Dsq[i] : 0.0, t.cs_w);
    t.Wm[i] = fx_const(w * o.Vq[i], t.cs_w);
  }
  for (int i = 0; i < NQ * NM; ++i) t.MP[i] = fx_const(mp[i], t.cs_m);
  for (int i = 0; i < NP * NP; ++i) t.Minv[i] = fx_const(o.Minv[i], t.cs_i);
  for (int m = 0; m < S::NFQ; ++m)
    for (int k = 0; k < S::NFP; ++k) t.LfT[k * S::NFQ + m] = fx_const(o.Lf[m * S::NFP + k], t.cs_w);
}

}  // namespace dgswe
