// Vector kernels of the point-block Jacobi PCG (ELAS3D-Xtal, arXiv 2602.07354, Algorithm 2).
//
// One iteration of Algorithm 2 is three launches on the device:
//   apply      Ah = A h with the h.Ah partial sums fused into its epilogue; a problem's last
//              item forms lambda = gg / hAh (step B) and applies the breakdown guard
//   update     g -= lambda Ah (step C), z = M^-1 g and gg = z.g, g.g (step D); a problem's last item
//              forms gg, gamma = gg / gg_last and decides convergence
//   direction  w -= lambda h (step C's other half) and h = z + gamma h (step E)
// w is advanced with the direction because that kernel reads h anyway: h is then read twice an
// iteration instead of three times, and the update's FP64 work falls by a seventh.  A solve that stops
// in its update, and every FP64 residual, brings w up to date first (k_w_finish).
// Every launch walks a flattened list of (problem, node chunk) items over all problems of the
// batch (one problem = one RVE with one load case).  All scalars live in device memory
// (DevState per problem), so a batch of iterations runs without the host; a finished (or
// paused) problem's items return at once.  Each item publishes its partial sums, and the
// problem's last item adds them in chunk order, so a problem's result is bitwise reproducible
// and independent of the other problems in the launch.
//
// Precision: the vector type Tv is double (FP64 path) or float (mixed path).  In the mixed path
// w is an unevaluated pair of floats updated with error-free transformations and the dot
// products accumulate compensated pairs, so no FP64 arithmetic runs per node (GB300 issues FP64
// at 1/64 of the FP32 rate).
#include <cuda_runtime.h>

#include "elas_internal.h"

namespace elas {

namespace {

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

__device__ double block_sum(double v, double* red) {
  v = warp_sum(v);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) red[wid] = v;
  __syncthreads();
  double r = 0.0;
  if (threadIdx.x == 0) {
    const int nw = (blockDim.x + 31) >> 5;
    for (int i = 0; i < nw; ++i) r += red[i];
  }
  return r;
}

__device__ double total_of(const double* slot, int n, double* red) {
  double v = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) v += __ldcg(slot + i);
  return block_sum(v, red);
}

// Publishes the partials this block has written; true in every thread of the problem's last item.
__device__ bool arrive_item(const Prob& P, unsigned int* ctr, int* s_last) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    *s_last = atomicAdd(ctr, 1u) == (unsigned)(P.n_vitems - 1);
  }
  __syncthreads();
  return *s_last != 0;
}

__device__ __forceinline__ int wrapi(int i, int n) {
  while (i < 0) i += n;
  while (i >= n) i -= n;
  return i;
}

template <typename Tv>
__device__ __forceinline__ void jacobi_apply(const Tv* __restrict__ minv, long long N, long long n, const Tv (&g)[3],
                                             Tv (&z)[3]) {
  const Tv m11 = minv[n], m22 = minv[N + n], m33 = minv[2 * N + n];
  const Tv m23 = minv[3 * N + n], m13 = minv[4 * N + n], m12 = minv[5 * N + n];
  z[0] = m11 * g[0] + m12 * g[1] + m13 * g[2];
  z[1] = m12 * g[0] + m22 * g[1] + m23 * g[2];
  z[2] = m13 * g[0] + m23 * g[1] + m33 * g[2];
}

// Solve setup per problem: tolerances, applied strain, counters; marks the problem for k_pcg_init.
__global__ void k_state_init(const Prob* __restrict__ probs, const SolveSetup* __restrict__ setups,
                             const int* __restrict__ idx, int n) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  DevState* st = probs[idx ? idx[k] : k].st;
  const SolveSetup s = setups[k];
  st->tol = s.tol;
  st->tol2_true = s.tol2_true;
  st->bscale2 = s.bscale2;
  st->max_iter = s.max_iter;
  st->stop_rule = s.stop_rule;
  st->replace_every = s.replace_every;
  st->drop2 = s.drop2;
  for (int q = 0; q < 9; ++q) st->E[q] = s.E[q];
  st->iter = 0;
  st->n_repl = 0;
  st->want_check = 0;
  st->last_repl_iter = 0;
  st->done = 0;
  st->needs_init = 1;
  st->finalized = 0;  // a server slot keeps its state: the request before this one has been finalised
  st->w_applied = 1;
  st->status = ST_RUNNING;
  st->gg = st->gg0 = st->gg_last = st->hAh = st->hAh_first = st->lambda = st->gamma = 0.0;
  st->rr = st->bb = st->rr_true = 0.0;
  for (int q = 0; q < 8; ++q) st->ctr[q] = 0u;  // in case an earlier solve ended inside a reduction
}

// Initial state of Algorithm 2 in fluctuation form: w = 0, g = b (right-hand side of Eqs. 7-8
// from the closed form b_m = sum_e sigma_e . s_a / 4), z = M^-1 g, h = z, gg0 = z.g.
template <typename Tv>
__global__ void k_pcg_init(const Prob* __restrict__ probs, const int* __restrict__ vitem_prob,
                           const long long* __restrict__ counts) {
  __shared__ double red[32];
  __shared__ int s_last;
  const long long n_items = counts[1];
  for (long long item = blockIdx.x; item < n_items; item += gridDim.x) {
    const Prob& P = probs[vitem_prob[item]];
    if (!P.st->needs_init) continue;  // only problems set up since their last start
    const long long N = P.N;
    const int nx = P.nx, ny = P.ny, nz = P.nz;
    Tv* __restrict__ g = reinterpret_cast<Tv*>(P.g);
    Tv* __restrict__ h = reinterpret_cast<Tv*>(P.h);
    Tv* __restrict__ z = reinterpret_cast<Tv*>(P.z);
    double* __restrict__ w = P.w;
    float* __restrict__ w_hi = P.w_hi;
    float* __restrict__ w_lo = P.w_lo;
    const int32_t* __restrict__ phase = P.phase;
    const double* __restrict__ sig = P.sig;
    const Tv* __restrict__ minv = reinterpret_cast<const Tv*>(P.minv);
    const int c0 = (int)(item - P.item0_vec) * P.vmerge, c1 = min(c0 + P.vmerge, P.n_chunks);
    for (int chunk = c0; chunk < c1; ++chunk) {
      const long long n0 = (long long)chunk * P.chunk, n1 = min(n0 + P.chunk, N);
      DotAcc<Tv> zg, gg2;
      DotAcc<double> bb;
      for (long long n = n0 + threadIdx.x; n < n1; n += kVecThreads) {
        const int i = (int)(n % nx), j = (int)((n / nx) % ny), k = (int)(n / ((long long)nx * ny));
        double b[3] = {0, 0, 0};
#pragma unroll
        for (int a = 0; a < 8; ++a) {
          const int ax = a & 1, ay = (a >> 1) & 1, az = (a >> 2) & 1;
          const long long e = (long long)wrapi(i - ax, nx) +
                              (long long)nx * (wrapi(j - ay, ny) + (long long)ny * wrapi(k - az, nz));
          const int ph = phase[e];
          if (ph < 0) continue;
          const double* S = sig + 6 * (long long)ph;
          const double sx = 0.25 * (2 * ax - 1), sy = 0.25 * (2 * ay - 1), sz = 0.25 * (2 * az - 1);
          b[0] += S[0] * sx + S[5] * sy + S[4] * sz;
          b[1] += S[5] * sx + S[1] * sy + S[3] * sz;
          b[2] += S[4] * sx + S[3] * sy + S[2] * sz;
        }
        Tv gv[3], zv[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          gv[c] = (Tv)b[c];
          bb.add(b[c], b[c]);
          gg2.add(gv[c], gv[c]);
        }
        jacobi_apply(minv, N, n, gv, zv);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          w[c * N + n] = 0.0;
          if (w_hi) {
            w_hi[c * N + n] = 0.f;
            w_lo[c * N + n] = 0.f;
          }
          g[c * N + n] = gv[c];
          z[c * N + n] = zv[c];
          h[c * N + n] = zv[c];
          zg.add(zv[c], gv[c]);
        }
      }
      const double vals[3] = {block_total(zg, red), block_total(bb, red), block_total(gg2, red)};
      if (threadIdx.x == 0)
        for (int q = 0; q < 3; ++q) P.parts[q * P.parts_stride + chunk] = vals[q];
    }
    if (arrive_item(P, &P.st->ctr[1], &s_last)) {
      const double s_zg = total_of(P.parts, P.n_chunks, red);
      const double s_bb = total_of(P.parts + P.parts_stride, P.n_chunks, red);
      const double s_gg = total_of(P.parts + 2 * P.parts_stride, P.n_chunks, red);
      if (threadIdx.x == 0) {
        DevState* st = P.st;
        st->ctr[1] = 0u;
        st->needs_init = 0;
        st->gg = st->gg0 = s_zg;
        st->bb = s_bb;
        st->rr = s_gg;
        st->rr_repl = s_gg;
        if (!isfinite(s_zg) || !isfinite(s_bb)) {
          st->status = ELAS_NONFINITE;
          st->done = 1;
        } else if (s_bb <= 1e-24 * st->bscale2) {
          // zero load (round-off of an exactly zero right-hand side): w = 0 is the solution
          st->status = ELAS_CONVERGED;
          st->done = 1;
        } else if (!(s_zg > 0.0)) {
          // z.g of a non-zero load is not positive: the preconditioner is not definite
          st->status = ELAS_BREAKDOWN;
          st->done = 1;
        } else if (st->max_iter <= 0) {
          st->status = ELAS_MAX_ITER;
          st->done = 1;
        }
      }
    }
    __syncthreads();
  }
}

// w -= lambda h for one component of one node.  Mixed path: w is the unevaluated pair (wh, wl), updated
// with error-free transformations (_rn intrinsics keep the compiler from contracting them into FMAs).
__device__ __forceinline__ void w_step(float& wh, float& wl, float h, float lam_hi, float lam_lo) {
  const float prod = __fmul_rn(lam_hi, h);
  const float perr = __fadd_rn(fmaf(lam_hi, h, -prod), __fmul_rn(lam_lo, h));  // lambda h = prod + perr
  const float s = __fsub_rn(wh, prod);  // two-sum of wh and -prod
  const float bb = __fsub_rn(s, wh);
  const float e = __fadd_rn(__fadd_rn(__fsub_rn(wh, __fsub_rn(s, bb)), __fsub_rn(-prod, bb)), __fsub_rn(wl, perr));
  const float nh = __fadd_rn(s, e);  // renormalise the pair
  wl = __fsub_rn(e, __fsub_rn(nh, s));
  wh = nh;
}

// One node of steps C and D without w: g -= lambda Ah, z = M^-1 g (symmetric inverse in Voigt slot
// order 11, 22, 33, 23, 13, 12), and the two dot terms.
template <typename Tv>
__device__ __forceinline__ void update_node(const Tv (&Ah)[3], Tv (&g)[3], const Tv (&m)[6], Tv (&z)[3], Tv lam,
                                            DotAcc<Tv>& zg, DotAcc<Tv>& gg2) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    g[c] = g[c] - lam * Ah[c];
    gg2.add(g[c], g[c]);
  }
  z[0] = m[0] * g[0] + m[5] * g[1] + m[4] * g[2];
  z[1] = m[5] * g[0] + m[1] * g[1] + m[3] * g[2];
  z[2] = m[4] * g[0] + m[3] * g[1] + m[2] * g[2];
#pragma unroll
  for (int c = 0; c < 3; ++c) zg.add(z[c], g[c]);
}

// The scalar step D/E of Algorithm 2 on a problem's totals z.g and g.g (one thread): gg,
// gamma = gg / gg_last, the iteration count and the stopping tests.
__device__ void update_scalar_step(DevState* st, double s_zg, double s_gg, bool mixed) {
  st->ctr[2] = 0u;
  st->gg_last = st->gg;
  st->gg = s_zg;
  st->rr = s_gg;
  st->iter += 1;
  st->w_applied = 0;  // the direction owes w its lambda h
  if (!isfinite(s_zg) || !isfinite(s_gg)) {
    st->status = ELAS_NONFINITE;
    st->done = 1;
  } else {
    const bool est = (st->stop_rule == ELAS_STOP_TRUE) ? (s_gg <= st->tol2_true * st->bb)
                                                        : (s_zg < st->tol * st->tol * st->gg0);
    if (est) {
      if (mixed || st->stop_rule == ELAS_STOP_TRUE) {
        st->want_check = 1;  // confirm on the FP64 true residual before stopping
      } else {
        st->status = ELAS_CONVERGED;
        st->done = 1;
      }
    } else if (st->iter >= st->max_iter) {
      st->status = ELAS_MAX_ITER;
      st->done = 1;
    }
    st->gamma = s_zg / st->gg_last;
    st->gam_f = (float)st->gamma;
  }
}

// Rows of consecutive nodes: 4 floats or 2 doubles (16 bytes), used for grids whose size is a multiple
// of the row (which path a node takes depends only on its problem).
template <typename Tv>
struct Row;
template <>
struct Row<float> {
  static constexpr int V = 4;
  using type = float4;
};
template <>
struct Row<double> {
  static constexpr int V = 2;
  using type = double2;
};
template <typename Tv, int V>
__device__ __forceinline__ void load_row(const Tv* __restrict__ p, Tv (&v)[V]) {
  if constexpr (V == 1)
    v[0] = *p;
  else
    *reinterpret_cast<typename Row<Tv>::type*>(v) = *reinterpret_cast<const typename Row<Tv>::type*>(p);
}
template <typename Tv, int V>
__device__ __forceinline__ void store_row(Tv* __restrict__ p, const Tv (&v)[V]) {
  if constexpr (V == 1)
    *p = v[0];
  else
    *reinterpret_cast<typename Row<Tv>::type*>(p) = *reinterpret_cast<const typename Row<Tv>::type*>(v);
}

template <typename Tv, int V>
__device__ __forceinline__ void update_chunk(const Prob& P, long long n0, long long n1, Tv lam, DotAcc<Tv>& zg,
                                             DotAcc<Tv>& gg2) {
  const long long N = P.N;
  Tv* __restrict__ gp = reinterpret_cast<Tv*>(P.g);
  const Tv* __restrict__ Ahp = reinterpret_cast<const Tv*>(P.Ah);
  Tv* __restrict__ zp = reinterpret_cast<Tv*>(P.z);
  const Tv* __restrict__ minv = reinterpret_cast<const Tv*>(P.minv);
  for (long long n = n0 + V * (int)threadIdx.x; n < n1; n += V * kVecThreads) {
    alignas(16) Tv A[3][V], g[3][V], m[6][V], z[3][V];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      load_row<Tv, V>(Ahp + c * N + n, A[c]);
      load_row<Tv, V>(gp + c * N + n, g[c]);
    }
#pragma unroll
    for (int q = 0; q < 6; ++q) load_row<Tv, V>(minv + q * N + n, m[q]);
#pragma unroll
    for (int j = 0; j < V; ++j) {
      const Tv Aj[3] = {A[0][j], A[1][j], A[2][j]}, mj[6] = {m[0][j], m[1][j], m[2][j], m[3][j], m[4][j], m[5][j]};
      Tv gj[3] = {g[0][j], g[1][j], g[2][j]}, zj[3];
      update_node(Aj, gj, mj, zj, lam, zg, gg2);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        g[c][j] = gj[c];
        z[c][j] = zj[c];
      }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      store_row<Tv, V>(gp + c * N + n, g[c]);
      store_row<Tv, V>(zp + c * N + n, z[c]);
    }
  }
}

// Step C's residual half and step D of Algorithm 2.  Each item publishes its partials (z.g, g.g); the
// problem's last item performs the scalar step.
template <typename Tv, bool ONE>
__device__ __forceinline__ void update_items(const Prob* __restrict__ probs, const int* __restrict__ vitem_prob,
                                             const long long* __restrict__ counts, const Prob& one) {
  __shared__ double buf[2 * kVecThreads];
  __shared__ int s_last;
  constexpr bool kMixed = sizeof(Tv) == 4;
  const long long n_items = ONE ? one.n_vitems : counts[1];
  for (long long item = blockIdx.x; item < n_items; item += gridDim.x) {
    const Prob& P = ONE ? one : probs[vitem_prob[item]];
    const DevState* cst = P.st;
    if (cst->done || cst->want_check) continue;
    const long long N = P.N;
    const Tv lam = kMixed ? (Tv)cst->lam_hi : (Tv)cst->lambda;
    const int V = N % Row<Tv>::V == 0 ? Row<Tv>::V : 1;
    const int c0 = (int)(item - P.item0_vec) * P.vmerge, c1 = ONE ? c0 + 1 : min(c0 + P.vmerge, P.n_chunks);
    for (int chunk = c0; chunk < c1; ++chunk) {
      const long long n0 = (long long)chunk * P.chunk, n1 = min(n0 + P.chunk, N);
      DotAcc<Tv> zg, gg2;
      if (V > 1)
        update_chunk<Tv, Row<Tv>::V>(P, n0, n1, lam, zg, gg2);
      else
        update_chunk<Tv, 1>(P, n0, n1, lam, zg, gg2);
      const double v = block_total2(zg, gg2, buf, min(kVecThreads, ((int)(n1 - n0) + V - 1) / V));
      if (threadIdx.x == 0) P.parts[chunk] = v;
      if (threadIdx.x == 32) P.parts[P.parts_stride + chunk] = v;
    }
    if (arrive_item(P, &P.st->ctr[2], &s_last)) {
      DotAcc<double> a, b;
      for (int i = threadIdx.x; i < P.n_chunks; i += kVecThreads) {
        a.s += __ldcg(P.parts + i);
        b.s += __ldcg(P.parts + P.parts_stride + i);
      }
      const double t = block_total2(a, b, buf, kVecThreads);
      if (threadIdx.x == 32) buf[kVecThreads] = t;  // (its readers are done: they are this warp)
      __syncthreads();
      if (threadIdx.x == 0) update_scalar_step(P.st, t, buf[kVecThreads], kMixed);
    }
    __syncthreads();
  }
}

// Bound: HBM and L2 for the rows (144 bytes a node in FP64, 72 mixed), the FP64 pipe (18 operations a
// node at 2 lanes per SM and clock) beside it in FP64.
// 100^3, with the direction: FP64 76 -> 63 us, mixed 37 -> 27 us an iteration (in the solve's graph).
template <bool ONE>
__global__ void __launch_bounds__(kVecThreads, 4)
    k_pcg_update_f64(const Prob* __restrict__ probs, const int* __restrict__ vitem_prob,
                     const long long* __restrict__ counts, const __grid_constant__ Prob one) {
  update_items<double, ONE>(probs, vitem_prob, counts, one);
}
template <bool ONE>
__global__ void __launch_bounds__(kVecThreads, 3)
    k_pcg_update_f32(const Prob* __restrict__ probs, const int* __restrict__ vitem_prob,
                     const long long* __restrict__ counts, const __grid_constant__ Prob one) {
  update_items<float, ONE>(probs, vitem_prob, counts, one);
}

// w -= lambda h and, with DIR, h = z + gamma h (step E, Fletcher-Reeves direction) on a chunk's nodes.
template <typename Tv, int V, bool DIR>
__device__ __forceinline__ void direction_chunk(const Prob& P, long long n0, long long n1, bool w_due, Tv gam) {
  const long long N = P.N;
  const DevState* st = P.st;
  const double lam = st->lambda;
  const float lam_hi = st->lam_hi, lam_lo = st->lam_lo;
  Tv* __restrict__ h = reinterpret_cast<Tv*>(P.h);
  const Tv* __restrict__ z = reinterpret_cast<const Tv*>(P.z);
  double* __restrict__ w = P.w;
  float* __restrict__ w_hi = P.w_hi;
  float* __restrict__ w_lo = P.w_lo;
  for (long long n = n0 + V * (int)threadIdx.x; n < n1; n += V * kVecThreads) {
    alignas(16) Tv hv[3][V], zv[3][V], a[3][V], b[3][V];  // a, b: w, or its pair
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      load_row<Tv, V>(h + c * N + n, hv[c]);
      if (DIR) load_row<Tv, V>(z + c * N + n, zv[c]);
      if (w_due) {
        if constexpr (sizeof(Tv) == 4) {
          load_row<Tv, V>(w_hi + c * N + n, a[c]);
          load_row<Tv, V>(w_lo + c * N + n, b[c]);
        } else {
          load_row<Tv, V>(w + c * N + n, a[c]);
        }
      }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      if (w_due) {
#pragma unroll
        for (int j = 0; j < V; ++j) {
          if constexpr (sizeof(Tv) == 4)
            w_step(a[c][j], b[c][j], hv[c][j], lam_hi, lam_lo);
          else
            a[c][j] -= lam * hv[c][j];
        }
        if constexpr (sizeof(Tv) == 4) {
          store_row<Tv, V>(w_hi + c * N + n, a[c]);
          store_row<Tv, V>(w_lo + c * N + n, b[c]);
        } else {
          store_row<Tv, V>(w + c * N + n, a[c]);
        }
      }
      if (DIR) {
#pragma unroll
        for (int j = 0; j < V; ++j) hv[c][j] = zv[c][j] + gam * hv[c][j];
        store_row<Tv, V>(h + c * N + n, hv[c]);
      }
    }
  }
}

// Bound: HBM and L2 (120 bytes a node in FP64, 84 mixed).
template <typename Tv, bool ONE>
__global__ void __launch_bounds__(kVecThreads, sizeof(Tv) == 8 ? 4 : 3)
    k_pcg_direction(const Prob* __restrict__ probs, const int* __restrict__ vitem_prob,
                    const long long* __restrict__ counts, const __grid_constant__ Prob one) {
  const long long n_items = ONE ? one.n_vitems : counts[1];
  for (long long item = blockIdx.x; item < n_items; item += gridDim.x) {
    const Prob& P = ONE ? one : probs[vitem_prob[item]];
    const DevState* cst = P.st;
    if (cst->done || cst->want_check) continue;
    const long long per = (long long)P.chunk * P.vmerge, n0 = (item - P.item0_vec) * per, n1 = min(n0 + per, P.N);
    const Tv gam = sizeof(Tv) == 4 ? (Tv)cst->gam_f : (Tv)cst->gamma;
    const bool w_due = !cst->w_applied;
    if (P.N % Row<Tv>::V == 0)
      direction_chunk<Tv, Row<Tv>::V, true>(P, n0, n1, w_due, gam);
    else
      direction_chunk<Tv, 1, true>(P, n0, n1, w_due, gam);
  }
}

// Brings w up to date: the pending w -= lambda h of a problem that stopped in its update or is about
// to have its residual replaced (a problem still running otherwise has had it from its direction),
// and in the mixed path w = w_hi + w_lo in FP64.  Gated like the kernel that follows it: the residual
// replacement, or the final true residual of a stopped problem.
template <typename Tv>
__global__ void __launch_bounds__(kVecThreads)
    k_w_finish(const Prob* __restrict__ probs, const int* __restrict__ vitem_prob, const long long* __restrict__ counts,
               int gate) {
  const long long n_items = counts[1];
  for (long long item = blockIdx.x; item < n_items; item += gridDim.x) {
    const Prob& P = probs[vitem_prob[item]];
    const DevState* st = P.st;
    if (gate == GATE_REPLACE && (st->done || !replacement_due(st))) continue;
    if (gate == GATE_FINALIZE && (!st->done || st->finalized)) continue;
    const long long N = P.N, per = (long long)P.chunk * P.vmerge;
    const long long n0 = (item - P.item0_vec) * per, n1 = min(n0 + per, N);
    if (!st->w_applied && (gate == GATE_REPLACE || st->done)) direction_chunk<Tv, 1, false>(P, n0, n1, true, Tv(0));
    if constexpr (sizeof(Tv) == 4) {  // a thread reads back its own nodes
      for (long long n = n0 + threadIdx.x; n < n1; n += kVecThreads)
#pragma unroll
        for (int c = 0; c < 3; ++c) P.w[c * N + n] = (double)P.w_hi[c * N + n] + (double)P.w_lo[c * N + n];
    }
  }
}

}  // namespace

cudaError_t launch_state_init(const BatchDev& b, const SolveSetup* setups, const int* idx, int n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_state_init<<<(n + 127) / 128, 128, 0, s>>>(b.probs, setups, idx, n);
  return cudaGetLastError();
}

cudaError_t launch_pcg_init(const BatchDev& b, bool mixed, cudaStream_t s) {
  if (mixed)
    k_pcg_init<float><<<b.vec_blocks, b.vec_threads, 0, s>>>(b.probs, b.vitem_prob, b.counts);
  else
    k_pcg_init<double><<<b.vec_blocks, b.vec_threads, 0, s>>>(b.probs, b.vitem_prob, b.counts);
  return cudaGetLastError();
}

// A batch of one problem passes its descriptor as an argument: its blocks start on their nodes
// without the chain of loads item -> problem -> pointers.
cudaError_t launch_pcg_update(const BatchDev& b, bool mixed, cudaStream_t s) {
  auto k = mixed ? (b.single ? k_pcg_update_f32<true> : k_pcg_update_f32<false>)
                 : (b.single ? k_pcg_update_f64<true> : k_pcg_update_f64<false>);
  k<<<b.vec_blocks, b.vec_threads, 0, s>>>(b.probs, b.vitem_prob, b.counts, b.one);
  return cudaGetLastError();
}

cudaError_t launch_pcg_direction(const BatchDev& b, bool mixed, cudaStream_t s) {
  auto k = mixed ? (b.single ? k_pcg_direction<float, true> : k_pcg_direction<float, false>)
                 : (b.single ? k_pcg_direction<double, true> : k_pcg_direction<double, false>);
  k<<<b.vec_blocks, b.vec_threads, 0, s>>>(b.probs, b.vitem_prob, b.counts, b.one);
  return cudaGetLastError();
}

cudaError_t launch_w_finish(const BatchDev& b, bool mixed, int gate, cudaStream_t s) {
  if (mixed)
    k_w_finish<float><<<b.vec_blocks, b.vec_threads, 0, s>>>(b.probs, b.vitem_prob, b.counts, gate);
  else
    k_w_finish<double><<<b.vec_blocks, b.vec_threads, 0, s>>>(b.probs, b.vitem_prob, b.counts, gate);
  return cudaGetLastError();
}

}  // namespace elas
