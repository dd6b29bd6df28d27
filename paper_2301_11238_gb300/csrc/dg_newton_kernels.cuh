// Kernels of the backward-Euler Newton-Krylov solver (dg_newton.h) that work on
// one element at a time.  Included by dg_kernels.cuh.
//
// A group of lanes shares an element, lane a its node a: a warp-wide FP64
// instruction takes 64 clocks whatever the lanes, so a thread per element would
// make the small meshes the solver is used on wait for one long chain.
// Tables come from shared memory, nodal values from the neighbouring lanes.
#pragma once

namespace dgswe {

// Lanes per element: the power of two that holds the nodes.
template <int DIM, int P>
constexpr int nk_lanes() {
  constexpr int NP = Sh<DIM, P>::NP;
  return NP <= 2 ? 2 : NP <= 4 ? 4 : NP <= 8 ? 8 : 16;
}
constexpr int kNkBlock = 128;

// l_a(q) and w_q l_a(q), then Minv.
template <int DIM, int P>
struct NkTab {
  static constexpr int NP = Sh<DIM, P>::NP, NQ = Sh<DIM, P>::NQ;
  double l[NQ * NP], wl[NQ * NP], Minv[NP * NP];
};
template <int DIM, int P>
__device__ __forceinline__ void nk_table(NkTab<DIM, P>& t, const VolOps<DIM, P, double>& ops) {
  using T = NkTab<DIM, P>;
  for (int i = threadIdx.x; i < T::NQ * T::NP; i += blockDim.x) {
    t.l[i] = ops.Vq[i];
    t.wl[i] = ops.Wm[i];
  }
  for (int i = threadIdx.x; i < T::NP * T::NP; i += blockDim.x) t.Minv[i] = ops.Minv[i];
  __syncthreads();
}

// Block sum of v in thread 0 (whole warps, fixed order); sh: one slot a warp.
__device__ __forceinline__ double block_sum_fixed(double v, double* sh) {
  v = warp_sum(v);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x < 32) t = warp_sum(threadIdx.x < (blockDim.x >> 5) ? sh[threadIdx.x] : 0.0);
  return t;
}
// Sums finished by the grid's last block: dot i is the sum of partial[i * G + b]
// over its G blocks, a warp a dot, in a fixed order.  counter is zero before and
// after.  Every thread of every block calls this after its block's partial has
// been written by thread 0.
__device__ __forceinline__ void finish_sums(int G, int cnt, const double* partial, double* out, unsigned* counter) {
  __shared__ bool last;
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(counter, 1u) == gridDim.x * gridDim.y - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int i = threadIdx.x >> 5; i < cnt; i += blockDim.x >> 5) {
    const double* p = partial + (size_t)i * G;
    // eight loads in flight a lane: their latency, not the additions, was the time
    double acc = 0.0;
    for (int b0 = threadIdx.x & 31; b0 < G; b0 += 256) {
      double v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = b0 + 32 * k < G ? __ldcg(p + b0 + 32 * k) : 0.0;
      acc += ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
    }
    acc = warp_sum(acc);
    if ((threadIdx.x & 31) == 0) out[i] = acc;
  }
  if (threadIdx.x == 0) *counter = 0;
}

// One element's group of lanes.
template <int DIM, int P>
struct NkLane {
  static constexpr int GL = nk_lanes<DIM, P>(), NP = Sh<DIM, P>::NP;
  int e, a;   // element (the last one for lanes past the end), node
  bool live;  // a node of an element
  __device__ explicit NkLane(int K, long long block = -1) {
    const long long g = (block < 0 ? (long long)blockIdx.x : block) * blockDim.x + threadIdx.x;
    const long long el = g / GL;
    a = (int)(g % GL);
    live = el < K && a < NP;
    e = (int)(el < K ? el : K - 1);
    if (a >= NP) a = NP - 1;
  }
};
template <int GL>
__device__ __forceinline__ double from_lane(double v, int src) {
  return __shfl_sync(0xffffffffu, v, src, GL);
}

// Nodal fields at the volume points q = lane, lane + GL, ..: at[i][v].
template <int DIM, int P>
__device__ __forceinline__ void nk_points(const double (&V)[Sh<DIM, P>::NV], const NkTab<DIM, P>& t, int lane,
                                          double (&at)[(Sh<DIM, P>::NQ + nk_lanes<DIM, P>() - 1) /
                                                       nk_lanes<DIM, P>()][Sh<DIM, P>::NV]) {
  using S = Sh<DIM, P>;
  constexpr int NP = S::NP, NQ = S::NQ, NV = S::NV, GL = nk_lanes<DIM, P>(), NS = (NQ + GL - 1) / GL;
#pragma unroll
  for (int i = 0; i < NS; ++i)
#pragma unroll
    for (int v = 0; v < NV; ++v) at[i][v] = 0.0;
#pragma unroll
  for (int b = 0; b < NP; ++b) {
    double x[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) x[v] = from_lane<GL>(V[v], b);
#pragma unroll
    for (int i = 0; i < NS; ++i) {
      const int q = min(lane + i * GL, NQ - 1);
      const double l = t.l[q * NP + b];
#pragma unroll
      for (int v = 0; v < NV; ++v) at[i][v] += l * x[v];
    }
  }
}

// <l_a, U_v(V)> per element in physical scaling, with U = (h, h u_1, ..,
// h u_d) (Eq. Uterm) at the volume quadrature points.  mode 0: out = that;
// mode 1: out += (that - Uold) * inv_dt, which adds the backward-Euler time
// term of Eq. WeakForm7 to the spatial residual already in out; mode 2: the
// directional difference of the residual so completed, out = (R - R0) / *eps.
template <int DIM, int P>
__global__ void __launch_bounds__(kNkBlock) be_time_kernel(int K, const double* __restrict__ V,
                                                           const double* __restrict__ Uold, double* __restrict__ out,
                                                           const double* __restrict__ geo,
                                                           const VolOps<DIM, P, double> ops, double inv_dt, int mode,
                                                           const double* __restrict__ R0,
                                                           const double* __restrict__ eps) {
  using S = Sh<DIM, P>;
  constexpr int NP = S::NP, NQ = S::NQ, NV = S::NV, GL = nk_lanes<DIM, P>(), NS = (NQ + GL - 1) / GL;
  __shared__ NkTab<DIM, P> t;
  nk_table<DIM, P>(t, ops);
  pdl_wait();
  pdl_trigger();
  after_wait(V, Uold, R0, eps);
  const NkLane<DIM, P> L(K);
  const size_t KN = (size_t)K * NP, o = (size_t)L.e * NP + L.a;
  double Vn[NV], at[NS][NV], acc[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    Vn[v] = V[v * KN + o];
    acc[v] = 0.0;
  }
  nk_points<DIM, P>(Vn, t, threadIdx.x % GL, at);
#pragma unroll
  for (int i = 0; i < NS; ++i)
#pragma unroll
    for (int v = 1; v < NV; ++v) at[i][v] *= at[i][0];
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const double wl = t.wl[q * NP + L.a];
#pragma unroll
    for (int v = 0; v < NV; ++v) acc[v] += wl * from_lane<GL>(at[q / GL][v], q % GL);
  }
  if (!L.live) return;
  const double J = geo[4 * (size_t)K + L.e];
  const double inv_eps = mode == 2 ? rcp_pos(*eps) : 0.0;
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const size_t i = v * KN + o;
    const double m = J * acc[v];
    if (mode == 0) {
      out[i] = m;
    } else {
      const double r = out[i] + (m - Uold[i]) * inv_dt;
      out[i] = mode == 1 ? r : (r - R0[i]) * inv_eps;
    }
  }
}

// Preconditioner dt M(V)^{-1} of the Newton-Krylov solve, M(V) the
// primitive-variable mass matrix (Appendix A, dU/dV).  V is fixed during a
// Krylov solve, so a Newton iteration forms, per element and in reference
// scaling, M_h^{-1} (Gauss-Jordan without pivoting: symmetric positive definite)
// and M_uj = <psi, u_j psi> once, and each application is three small
// matrix-vector products.  mats: [1 + DIM][K][NP][NP].
template <int DIM, int P>
__global__ void __launch_bounds__(kNkBlock) mass_factor_kernel(int K, const double* __restrict__ V,
                                                               double* __restrict__ mats,
                                                               const VolOps<DIM, P, double> ops, double h_floor) {
  using S = Sh<DIM, P>;
  constexpr int NP = S::NP, NQ = S::NQ, NV = S::NV, GL = nk_lanes<DIM, P>(), NS = (NQ + GL - 1) / GL;
  __shared__ NkTab<DIM, P> t;
  nk_table<DIM, P>(t, ops);
  pdl_wait();
  pdl_trigger();
  after_wait(V);
  const NkLane<DIM, P> L(K);
  const size_t KN = (size_t)K * NP, o = (size_t)L.e * NP + L.a;
  double Vn[NV], at[NS][NV], M[NV][NP];  // row a of M_h, M_u1, ..
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    Vn[v] = V[v * KN + o];
#pragma unroll
    for (int b = 0; b < NP; ++b) M[v][b] = 0.0;
  }
  nk_points<DIM, P>(Vn, t, threadIdx.x % GL, at);
#pragma unroll
  for (int i = 0; i < NS; ++i) at[i][0] = max_pos(at[i][0], h_floor);
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const double wl = t.wl[q * NP + L.a];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const double x = wl * from_lane<GL>(at[q / GL][v], q % GL);
#pragma unroll
      for (int b = 0; b < NP; ++b) M[v][b] += x * t.l[q * NP + b];
    }
  }
#pragma unroll
  for (int k = 0; k < NP; ++k) {
    double p[NP];
#pragma unroll
    for (int b = 0; b < NP; ++b) p[b] = from_lane<GL>(M[0][b], k);
    const double inv = rcp_pos(p[k]);
    const bool own = threadIdx.x % GL == k;
    const double f = M[0][k] * inv;
#pragma unroll
    for (int b = 0; b < NP; ++b) {
      if (b == k) M[0][b] = own ? inv : -f;
      else M[0][b] = own ? p[b] * inv : M[0][b] - f * p[b];
    }
  }
  if (!L.live) return;
#pragma unroll
  for (int v = 0; v < NV; ++v)
#pragma unroll
    for (int b = 0; b < NP; ++b) mats[((v * (size_t)K + L.e) * NP + b) * NP + L.a] = M[v][b];
}

// z = scale M(V)^{-1} x.  nrm2 given: x is divided by sqrt(*nrm2) first and
// written to xn.  add: z is added to out instead of stored; otherwise *zz = <z, z>
// (partial: one slot a block).  Blocks of lane groups in a grid-stride loop.
template <int DIM, int P>
__global__ void __launch_bounds__(kNkBlock) mass_apply_kernel(int K, const double* __restrict__ x,
                                                              const double* __restrict__ mats,
                                                              const double* __restrict__ geo,
                                                              const VolOps<DIM, P, double> ops, double scale,
                                                              const double* __restrict__ nrm2,
                                                              double* __restrict__ xn, double* __restrict__ out,
                                                              int add, double* partial, double* zz,
                                                              unsigned* counter) {
  using S = Sh<DIM, P>;
  constexpr int NP = S::NP, NV = S::NV, GL = nk_lanes<DIM, P>();
  __shared__ NkTab<DIM, P> t;
  nk_table<DIM, P>(t, ops);
  pdl_wait();
  pdl_trigger();
  after_wait(x, mats, nrm2);
  const size_t KN = (size_t)K * NP;
  const double nrm = nrm2 ? 1.0 / sqrt(*nrm2) : 1.0;
  const long long blocks = ((long long)K * GL + kNkBlock - 1) / kNkBlock;
  double acc = 0.0;
  for (long long blk = blockIdx.x; blk < blocks; blk += gridDim.x) {
    const NkLane<DIM, P> L(K, blk);
    const size_t o = (size_t)L.e * NP + L.a;
    const double Jinv = geo[6 * (size_t)K + L.e];
    double xr[NV], z[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      xr[v] = nrm * x[v * KN + o];
      if (nrm2 && L.live) xn[v * KN + o] = xr[v];
      xr[v] *= Jinv;
    }
    z[0] = 0.0;
#pragma unroll
    for (int b = 0; b < NP; ++b) z[0] += t.Minv[L.a * NP + b] * from_lane<GL>(xr[0], b);
#pragma unroll
    for (int j = 1; j < NV; ++j) {
#pragma unroll
      for (int b = 0; b < NP; ++b)
        xr[j] -= mats[((j * (size_t)K + L.e) * NP + b) * NP + L.a] * from_lane<GL>(z[0], b);
      z[j] = 0.0;
    }
#pragma unroll
    for (int b = 0; b < NP; ++b) {
      const double m = mats[((size_t)L.e * NP + b) * NP + L.a];
#pragma unroll
      for (int j = 1; j < NV; ++j) z[j] += m * from_lane<GL>(xr[j], b);
    }
    if (L.live) {
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const size_t i = v * KN + o;
        const double y = scale * z[v];
        out[i] = add ? out[i] + y : y;
        acc += y * y;
      }
    }
  }
  if (add) return;
  __shared__ double sh[kNkBlock / 32];
  acc = block_sum_fixed(acc, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = acc;
  finish_sums(gridDim.x, 1, partial, zz, counter);
}

}  // namespace dgswe
