// Microstructure generator on the device (ELAS3D-Xtal, arXiv 2602.07354, Sec. 2.2): grain
// assignment by the weighted ellipsoidal distance of Algorithm 4 and the pore overwrite of
// Algorithm 5 (with rotated ellipsoids as well as spheres), on a periodic cell.
//
// Grain assignment: the seeds are binned on the host into a uniform grid of cells (about one seed
// per cell, like the coarse cell grid of the paper's seeding stage) and uploaded in cell order.  A
// block takes a tile of 8 x 8 x 8 voxels, collects the seeds of the cells around it, keeps those
// whose distance can reach below the smallest upper bound over the tile (typically 15-25 of a few
// hundred) and scans them in FP32; a voxel whose two best FP32 distances are further apart than
// twice the FP32 error bound has its grain, the few others compare their close candidates in FP64.
// D^2 is evaluated there with explicitly rounded FP64 operations in the order
// (dx*dx + dy*dy) / (rt*rt) + (dz*dz) / (rl*rl), with the periodic minimum-image differences, and
// ties go to the lowest grain index: every voxel gets exactly the grain of a brute-force scan.
//
// Pore overwrite: several blocks per pore scan the pore's bounding box (periodically wrapped) and
// write -1 into every voxel whose centre satisfies (q0/a0)^2 + (q1/a1)^2 + (q2/a2)^2 <= 1 with
// q = R^T d; the writes are idempotent, so the order of pores and threads does not matter.
#include <cuda_runtime.h>

#include <cmath>
#include <string>
#include <vector>

#include "elas_internal.h"

namespace elas {

namespace {

thread_local std::string g_gen_err;

constexpr int kGenWin = 2;         // cells scanned on each side of a voxel's own cell
constexpr int kGenMaxCells = 128;  // per dimension
constexpr int kGenThreads = 256;
constexpr int kPoreDoubles = 15;

int gen_fail(int code, const std::string& m) {
  g_gen_err = m;
  return code;
}

struct GenGrid {
  int g[3];        // cells per dimension
  double cs[3];    // cell size per dimension
  double inv_rmax2;  // 1 / (largest semi-axis)^2
};

GenGrid gen_grid(int nx, int ny, int nz, int n) {
  GenGrid G{};
  const double L[3] = {(double)nx, (double)ny, (double)nz};
  const double target = std::cbrt(L[0] * L[1] * L[2] / std::max(n, 1));  // ~1 seed per cell
  for (int d = 0; d < 3; ++d) {
    G.g[d] = (int)std::lround(L[d] / target);
    G.g[d] = std::max(1, std::min(kGenMaxCells, G.g[d]));
    G.cs[d] = L[d] / G.g[d];
  }
  return G;
}

struct GenLayout {
  size_t seeds, semi, fast, start, items, pores, counter, total;
};

GenLayout gen_layout(const GenGrid& G, int n_grains, int n_pores) {
  GenLayout L{};
  size_t o = 0;
  auto take = [&](size_t b) {
    const size_t at = o;
    o = (o + b + 255) / 256 * 256;
    return at;
  };
  const size_t cells = (size_t)G.g[0] * G.g[1] * G.g[2];
  L.seeds = take(sizeof(double) * 3 * std::max(n_grains, 1));
  L.semi = take(sizeof(double) * 2 * std::max(n_grains, 1));
  L.fast = take(sizeof(float4) * 2 * std::max(n_grains, 1));
  L.start = take(sizeof(int) * (cells + 1));
  L.items = take(sizeof(int) * std::max(n_grains, 1));
  L.pores = take(sizeof(double) * kPoreDoubles * std::max(n_pores, 1));
  L.counter = take(sizeof(unsigned long long) * 2);
  L.total = o;
  return L;
}

__device__ __forceinline__ double min_image(double d, double L) {
  if (d > 0.5 * L) return d - L;
  if (d < -0.5 * L) return d + L;
  return d;
}

// Algorithm 4's weighted ellipsoidal distance, rounded operation by operation.  Without weights
// (rt = rl = 1) the two divisions by 1 are exact and are left out.
template <bool WEIGHTED>
__device__ __forceinline__ double wdist2(const double (&x)[3], const double* __restrict__ s,
                                         const double* __restrict__ semi, int l, const double (&L)[3]) {
  const double dx = min_image(x[0] - s[0], L[0]);
  const double dy = min_image(x[1] - s[1], L[1]);
  const double dz = min_image(x[2] - s[2], L[2]);
  if (!WEIGHTED) return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
  const double rt = semi[2 * l], rl = semi[2 * l + 1];
  return __dadd_rn(__ddiv_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(rt, rt)),
                   __ddiv_rn(__dmul_rn(dz, dz), __dmul_rn(rl, rl)));
}

__device__ __forceinline__ void consider(double D2, int l, double& best, int& arg) {
  if (D2 < best || (D2 == best && l < arg)) {
    best = D2;
    arg = l;
  }
}

// The grain of one voxel by FP64 distances alone: the 5 x 5 x 5 cells around its own, and every seed
// when those cannot be shown to hold the nearest one (seeds outside that block lie at least the
// distance from the voxel to the block's faces away).  Tiles whose candidates do not fit the block's
// list and grids outside the FP32 screen's range (k_assign_exact) take it.
template <bool WEIGHTED>
__device__ int nearest_exact(const double (&x)[3], const double* __restrict__ seeds, const double* __restrict__ semi,
                             int n, const int* __restrict__ start, const int* __restrict__ items, const GenGrid& G,
                             const double (&L)[3]) {
  int c[3], lo[3], cnt[3];
  bool all[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    c[d] = min(G.g[d] - 1, max(0, (int)floor(x[d] / G.cs[d])));
    all[d] = G.g[d] <= 2 * kGenWin + 1;
    lo[d] = all[d] ? 0 : c[d] - kGenWin;
    cnt[d] = all[d] ? G.g[d] : 2 * kGenWin + 1;
  }
  double best = INFINITY;
  int arg = 0x7fffffff;
  for (int oz = 0; oz < cnt[2]; ++oz) {
    int cz = lo[2] + oz;
    cz += cz < 0 ? G.g[2] : (cz >= G.g[2] ? -G.g[2] : 0);
    for (int oy = 0; oy < cnt[1]; ++oy) {
      int cy = lo[1] + oy;
      cy += cy < 0 ? G.g[1] : (cy >= G.g[1] ? -G.g[1] : 0);
      for (int ox = 0; ox < cnt[0]; ++ox) {
        int cx = lo[0] + ox;
        cx += cx < 0 ? G.g[0] : (cx >= G.g[0] ? -G.g[0] : 0);
        const int cell = cx + G.g[0] * (cy + G.g[1] * cz);
        for (int t = start[cell]; t < start[cell + 1]; ++t)
          consider(wdist2<WEIGHTED>(x, seeds + 3 * t, semi, t, L), items[t], best, arg);
      }
    }
  }
  // every seed outside the scanned block is at least lb away (Euclidean) in some dimension
  double lb = INFINITY;
#pragma unroll
  for (int d = 0; d < 3; ++d)
    if (!all[d]) lb = fmin(lb, fmin(x[d] - (c[d] - kGenWin) * G.cs[d], (c[d] + kGenWin + 1) * G.cs[d] - x[d]));
  if (!(best < 0.999999 * lb * lb * G.inv_rmax2))
    for (int t = 0; t < n; ++t) consider(wdist2<WEIGHTED>(x, seeds + 3 * t, semi, t, L), items[t], best, arg);
  return arg;
}

// Every voxel by FP64 distances, one a thread (by tiles of k_assign, two a thread one after the other, 55
// seeds on 48^3 took 704 us, this form 545).
template <bool WEIGHTED>
__global__ void k_assign_exact(int nx, int ny, int nz, const double* __restrict__ seeds, const double* __restrict__ semi,
                               int n, const int* __restrict__ start, const int* __restrict__ items, GenGrid G,
                               int32_t* __restrict__ phase) {
  const long long N = (long long)nx * ny * nz;
  const double L[3] = {(double)nx, (double)ny, (double)nz};
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < N; v += (long long)gridDim.x * blockDim.x) {
    const double x[3] = {(int)(v % nx) + 0.5, (int)((v / nx) % ny) + 0.5, (int)(v / ((long long)nx * ny)) + 0.5};
    phase[v] = nearest_exact<WEIGHTED>(x, seeds, semi, n, start, items, G, L);
  }
}

// One tile of 8 x 8 x 8 voxels per block and turn, two voxels (z and z + 4) per thread.
//
// FP32 error.  A seed comes as a float pair hi + lo; its minimum-image offset from the tile's centre
// is o = (hi - c) + lo with c a half-integer (exact), so o is off by 2^-23 |o| at most.  With h the
// tile's half-edge a component of the voxel-seed difference, folded once more, is off by less than
// 2^-24 (5 |dx| + 2 h), and the weighted squared distance by less than 2^-19 (D^2 + 3 h^2 w), w the
// larger weight (weights are (rmax / r)^2 >= 1, rounded once).  Two seeds whose FP32 distances
// differ by more than 2^-17 (D^2 + 3 h^2 w) are therefore in the same order in FP64.
//
// Bound: the FP64 pipe when every candidate was compared in FP64 (125 seeds x ~10 operations a
// voxel: 39 ms for 160^3 voxels and 2,048 grains, pipe 85% busy); the pruned FP32 scan takes
// 0.096 ms, no FP64 left outside the few near ties.  Forming the offsets in FP64 (12
// operations a collected seed) took 206 us.
constexpr int kTile = 8, kTileCap = 4 * kGenThreads;
template <bool WEIGHTED>
__global__ void __launch_bounds__(kGenThreads)
    k_assign(int nx, int ny, int nz, const double* __restrict__ seeds, const double* __restrict__ semi,
             const float4* __restrict__ fast, int n, const int* __restrict__ start, const int* __restrict__ items,
             GenGrid G, int32_t* __restrict__ phase) {
  __shared__ float4 cand[kTileCap];                // offset from the tile's centre, seed position
  __shared__ float2 candw[WEIGHTED ? kTileCap : 1];  // transverse and longitudinal weights
  __shared__ int s_raw, s_cnt, s_ub, s_wmax, s_wrap, s_lo[3], s_n[3];
  __shared__ float s_c[3], s_h[3], s_margin[3];
  const int tid = threadIdx.x;
  const int n3[3] = {nx, ny, nz};
  const double L[3] = {(double)nx, (double)ny, (double)nz};
  const float Lf[3] = {(float)nx, (float)ny, (float)nz};
  const int tx = (nx - 1) / kTile + 1, ty = (ny - 1) / kTile + 1, tz = (nz - 1) / kTile + 1;
  const long long n_tiles = (long long)tx * ty * tz;
  const int i = tid % kTile, j = (tid / kTile) % kTile, k = tid / (kTile * kTile);  // and k + 4
  for (long long tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    const int org[3] = {(int)(tile % tx) * kTile, (int)((tile / tx) % ty) * kTile,
                        (int)(tile / ((long long)tx * ty)) * kTile};
    // the tile's centre, half-edges and cell window, one dimension per thread: FP64 divisions by every
    // thread would cost more FP64-pipe time than everything else here
    if (tid < 3) {
      const int d = tid;
      const double x0 = org[d] + 0.5, x1 = (n3[d] - org[d] > kTile ? org[d] + kTile : n3[d]) - 0.5;
      s_c[d] = (float)(0.5 * (x0 + x1));
      s_h[d] = (float)(0.5 * (x1 - x0));
      int l = min(G.g[d] - 1, (int)floor(x0 / G.cs[d])) - kGenWin;
      int m = min(G.g[d] - 1, (int)floor(x1 / G.cs[d])) + kGenWin - l + 1;
      s_margin[d] = (float)fmin(x0 - l * G.cs[d], (l + m) * G.cs[d] - x1);
      if (m >= G.g[d]) {
        l = 0;
        m = G.g[d];
        s_margin[d] = INFINITY;
      }
      s_lo[d] = l;
      s_n[d] = m;
    }
    if (tid == 0) {
      s_raw = s_cnt = s_wrap = 0;
      s_ub = __float_as_int(INFINITY);
      s_wmax = __float_as_int(1.f);
    }
    __syncthreads();
    const float cf[3] = {s_c[0], s_c[1], s_c[2]};
    const float h[3] = {s_h[0], s_h[1], s_h[2]}, margin = fminf(s_margin[0], fminf(s_margin[1], s_margin[2]));
    const int lo[3] = {s_lo[0], s_lo[1], s_lo[2]}, cnt[3] = {s_n[0], s_n[1], s_n[2]};
    const float hm = fmaxf(h[0], fmaxf(h[1], h[2])), h2 = 3.f * hm * hm;
    // seed t: its offset from the tile's centre, weights, and bounds of its distance over the tile
    auto bounds = [&](int t, float (&o)[3], float2& w, float& dlo, float& dhi) {
      const float4 hi = fast[2 * t], rest = fast[2 * t + 1];
      const float sh[3] = {hi.x, hi.y, hi.z}, sl[3] = {rest.x, rest.y, rest.z};
      float a[3], b[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        // (an offset within rounding of L / 2 may keep either sign: the scan folds differences again)
        o[d] = (sh[d] - cf[d]) + sl[d];
        if (fabsf(o[d]) > 0.5f * Lf[d]) o[d] = (sh[d] - (cf[d] + (o[d] > 0.f ? Lf[d] : -Lf[d]))) + sl[d];
        const float m = fabsf(o[d]);
        a[d] = fmaxf(0.f, m - h[d]);
        b[d] = fminf(m + h[d], 0.5f * Lf[d]);
      }
      w = WEIGHTED ? make_float2(hi.w, rest.w) : make_float2(1.f, 1.f);
      dlo = (a[0] * a[0] + a[1] * a[1]) * w.x + a[2] * a[2] * w.y;
      dhi = (b[0] * b[0] + b[1] * b[1]) * w.x + b[2] * b[2] * w.y;
    };
    bool all = false;
    auto each_seed = [&](auto&& f) {
      if (all) {
        for (int t = tid; t < n; t += kGenThreads) f(t);
        return;
      }
      // a row of cells along x is one or (wrapped) two runs of the sorted seeds; 8 lanes take a row
      for (int q = tid / 8; q < cnt[1] * cnt[2]; q += kGenThreads / 8) {
        int cy = lo[1] + q % cnt[1], cz = lo[2] + q / cnt[1];
        cy += cy < 0 ? G.g[1] : (cy >= G.g[1] ? -G.g[1] : 0);
        cz += cz < 0 ? G.g[2] : (cz >= G.g[2] ? -G.g[2] : 0);
        const int* row = start + (long long)G.g[0] * (cy + (long long)G.g[1] * cz);
        const int x0 = max(lo[0], 0), x1 = min(lo[0] + cnt[0], G.g[0]);
        const int end = row[x1];
        for (int t = row[x0] + tid % 8; t < end; t += 8) f(t);
        const int w0 = lo[0] < 0 ? lo[0] + G.g[0] : 0, w1 = lo[0] < 0 ? G.g[0] : lo[0] + cnt[0] - G.g[0];
        if (w1 > w0) {
          const int wend = row[w1];
          for (int t = row[w0] + tid % 8; t < wend; t += 8) f(t);
        }
      }
    };
    float ub;
    // the smallest upper bound over the tile; the candidates wait in the list as they come
    for (int pass = 0; pass < 2; ++pass) {
      float mine = INFINITY;
      each_seed([&](int t) {
        float o[3], dlo, dhi;
        float2 w;
        bounds(t, o, w, dlo, dhi);
        mine = fminf(mine, dhi);
        const int at = atomicAdd(&s_raw, 1);
        if (at < kTileCap) {
          cand[at] = make_float4(o[0], o[1], o[2], __int_as_float(t));
          if (WEIGHTED) candw[at] = w;
        }
      });
#pragma unroll
      for (int s = 16; s > 0; s >>= 1) mine = fminf(mine, __shfl_xor_sync(0xffffffffu, mine, s));
      if ((tid & 31) == 0) atomicMin(&s_ub, __float_as_int(mine));  // non-negative floats order as ints
      __syncthreads();
      ub = __int_as_float(s_ub);
      // a seed outside the collected cells is at least the margin away, at weight >= 1
      if (pass == 1 || ub < 0.999f * margin * margin) break;
      all = true;
      __syncthreads();
      if (tid == 0) s_raw = 0;
      __syncthreads();
    }
    // the largest lower bound that a seed of these weights may have and still win a voxel.  A lower bound
    // is off by 2^-21 (D^2 + 3 h^2 w) at most: the rounding of an offset is 2^-23 (a + h) and enters 2 a w
    // times (without w in it, a seed of weight 1e8 just outside a tile lost voxels that were its own)
    auto reach = [&](const float2& w) { return ub + 1e-4f * (ub + h2 * fmaxf(w.x, w.y)); };
    const int raw = s_raw;
    auto wraps = [&](float ox, float oy, float oz) {
      return fabsf(ox) + h[0] > 0.499f * Lf[0] || fabsf(oy) + h[1] > 0.499f * Lf[1] || fabsf(oz) + h[2] > 0.499f * Lf[2];
    };
    auto keep = [&](const float4& v, const float2& w) {
      const int at = atomicAdd(&s_cnt, 1);
      if (at < kTileCap) {
        cand[at] = v;
        if (WEIGHTED) candw[at] = w;
      }
      if (wraps(v.x, v.y, v.z)) s_wrap = 1;
      if (WEIGHTED) atomicMax(&s_wmax, __float_as_int(fmaxf(w.x, w.y)));
    };
    if (raw <= kTileCap) {  // compact the list in place
      float4 v[4];
      float2 w[4];
      bool in[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int at = tid + q * kGenThreads;
        in[q] = at < raw;
        if (in[q]) {
          v[q] = cand[at];
          w[q] = WEIGHTED ? candw[at] : make_float2(1.f, 1.f);
          const float a = fmaxf(0.f, fabsf(v[q].x) - h[0]), b = fmaxf(0.f, fabsf(v[q].y) - h[1]);
          const float e = fmaxf(0.f, fabsf(v[q].z) - h[2]);
          in[q] = (a * a + b * b) * w[q].x + e * e * w[q].y <= reach(w[q]);
        }
      }
      __syncthreads();
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (in[q]) keep(v[q], w[q]);
    } else {  // more candidates than the list holds: collect again, pruned
      __syncthreads();
      each_seed([&](int t) {
        float o[3], dlo, dhi;
        float2 w;
        bounds(t, o, w, dlo, dhi);
        if (dlo <= reach(w)) keep(make_float4(o[0], o[1], o[2], __int_as_float(t)), w);
      });
    }
    __syncthreads();
    const int m = s_cnt;
    const int vi = org[0] + i, vj = org[1] + j;
    const bool in_xy = vi < nx && vj < ny;
    if (m <= kTileCap) {
      const float rx = (float)i - h[0], ry = (float)j - h[1], rz[2] = {(float)k - h[2], (float)(k + 4) - h[2]};
      const bool wrap = s_wrap != 0;
      float m1[2] = {INFINITY, INFINITY}, m2[2] = {INFINITY, INFINITY};
      int arg[2] = {0, 0};
      auto dist = [&](int q, float (&D)[2], int& t) {
        const float4 v = cand[q];
        t = __float_as_int(v.w);
        float a = fabsf(rx - v.x), b = fabsf(ry - v.y), e0 = fabsf(rz[0] - v.z), e1 = fabsf(rz[1] - v.z);
        if (wrap) {
          a = fminf(a, Lf[0] - a);
          b = fminf(b, Lf[1] - b);
          e0 = fminf(e0, Lf[2] - e0);
          e1 = fminf(e1, Lf[2] - e1);
        }
        float xy = fmaf(a, a, b * b);
        if (WEIGHTED) {
          const float2 w = candw[q];
          xy *= w.x;
          D[0] = fmaf(e0 * e0, w.y, xy);
          D[1] = fmaf(e1 * e1, w.y, xy);
        } else {
          D[0] = fmaf(e0, e0, xy);
          D[1] = fmaf(e1, e1, xy);
        }
      };
      for (int q = 0; q < m; ++q) {
        float D[2];
        int t;
        dist(q, D, t);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          m2[s] = fminf(m2[s], fmaxf(m1[s], D[s]));
          if (D[s] < m1[s]) arg[s] = t;
          m1[s] = fminf(m1[s], D[s]);
        }
      }
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        const int vk = org[2] + k + 4 * s;
        if (!in_xy || vk >= nz) continue;
        int id;
        const float T = m1[s] + 0x1p-17f * (m1[s] + h2 * __int_as_float(s_wmax));
        if (m2[s] > T) {
          id = items[arg[s]];
        } else {
          const double x[3] = {vi + 0.5, vj + 0.5, vk + 0.5};
          double best = INFINITY;
          id = 0x7fffffff;
          for (int q = 0; q < m; ++q) {
            float D[2];
            int t;
            dist(q, D, t);
            if (D[s] <= T) consider(wdist2<WEIGHTED>(x, seeds + 3 * t, semi, t, L), items[t], best, id);
          }
        }
        phase[vi + (long long)nx * (vj + (long long)ny * vk)] = id;
      }
    } else {
#pragma unroll 1
      for (int s = 0; s < 2; ++s) {
        const int vk = org[2] + k + 4 * s;
        if (!in_xy || vk >= nz) continue;
        const double x[3] = {vi + 0.5, vj + 0.5, vk + 0.5};
        phase[vi + (long long)nx * (vj + (long long)ny * vk)] =
            nearest_exact<WEIGHTED>(x, seeds, semi, n, start, items, G, L);
      }
    }
    __syncthreads();  // the list is reused by the next tile
  }
}

// Several blocks per pore (blockIdx.y) share its bounding box.  The membership sum is formed in FP32
// first.  With |R_ij| <= 1 (to rounding), semi-axes within a factor 20 of each other and
// amax >= 1/2, a difference is at most amax + 3 long inside the box, so u = R^T d / a is off by less
// than 1e-4 and the sum by less than 4e-4 of max(1, sum): only voxels within 1e-3 of the surface
// evaluate the FP64 sum, and voxels with a component within 1e-6 of half the cell, where rounding may pick
// the other minimum image (a frame that is not a rotation may have either image inside).
// Bound: FP64 arithmetic before (183 pores of r <= 6: 71 us with R / a still divided in FP64 by every
// thread); 12.7 us now, issue-bound.
__global__ void k_stamp(int nx, int ny, int nz, const double* __restrict__ pores, int32_t* __restrict__ phase) {
  const double* P = pores + (size_t)kPoreDoubles * blockIdx.x;
  __shared__ float sP[kPoreDoubles], s_first[3];
  __shared__ int s_lo[3], s_ext;
  const int n[3] = {nx, ny, nz};
  if (threadIdx.x < kPoreDoubles) sP[threadIdx.x] = (float)P[threadIdx.x];
  if (threadIdx.x < 3) {
    const int d = threadIdx.x, ext = (int)ceil(fmax(P[3], fmax(P[4], P[5]))) + 1;
    const int l = 2 * ext + 1 >= n[d] ? 0 : (int)floor(P[d]) - ext;
    s_lo[d] = l;
    s_first[d] = (float)(l + 0.5 - P[d]);
    if (d == 0) s_ext = ext;
  }
  __syncthreads();
  int lo[3], cnt[3];
  float first[3], Q[9], rmax = 0.f;  // Q = R / a
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    lo[d] = s_lo[d];
    cnt[d] = min(2 * s_ext + 1, n[d]);
    first[d] = s_first[d];
  }
#pragma unroll
  for (int q = 0; q < 9; ++q) {
    rmax = fmaxf(rmax, fabsf(sP[6 + q]));
    Q[q] = sP[6 + q] / sP[3 + q % 3];
  }
  const float amax = fmaxf(sP[3], fmaxf(sP[4], sP[5]));
  const bool screen = rmax <= 1.001f && amax >= 0.5f && amax < 1e4f && fminf(sP[3], fminf(sP[4], sP[5])) >= 0.05f * amax;
  const unsigned total = (unsigned)cnt[0] * cnt[1] * cnt[2];
  for (unsigned t = blockIdx.y * blockDim.x + threadIdx.x; t < total; t += gridDim.y * blockDim.x) {
    const int at[3] = {(int)(t % cnt[0]), (int)((t / cnt[0]) % cnt[1]), (int)(t / ((unsigned)cnt[0] * cnt[1]))};
    int idx[3];
    float f[3];
    bool half = false;  // half a cell away but for rounding (1.5e-7 of the cell)
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const int a = lo[d] + at[d];  // -n < a < 2 n
      idx[d] = a < 0 ? a + n[d] : (a >= n[d] ? a - n[d] : a);
      f[d] = first[d] + (float)at[d];
      const float Lf = (float)n[d];
      f[d] -= f[d] > 0.5f * Lf ? Lf : (f[d] < -0.5f * Lf ? -Lf : 0.f);
      half = half || fabsf(fabsf(f[d]) - 0.5f * Lf) <= 1e-6f * Lf;
    }
    float sf = 0.f;
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const float u = Q[m] * f[0] + Q[3 + m] * f[1] + Q[6 + m] * f[2];
      sf = fmaf(u, u, sf);
    }
    bool inside = sf < 1.f;
    if (!screen || half || !(fabsf(sf - 1.f) > 1e-3f * fmaxf(1.f, sf))) {
      double dd[3], s = 0.0;
#pragma unroll
      for (int d = 0; d < 3; ++d) dd[d] = min_image(idx[d] + 0.5 - P[d], (double)n[d]);
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        const double q = __dadd_rn(__dadd_rn(__dmul_rn(P[6 + m], dd[0]), __dmul_rn(P[9 + m], dd[1])), __dmul_rn(P[12 + m], dd[2]));
        const double u = __ddiv_rn(q, P[3 + m]);
        s = __dadd_rn(s, __dmul_rn(u, u));
      }
      inside = s <= 1.0;
    }
    if (inside) phase[idx[0] + (long long)nx * (idx[1] + (long long)ny * idx[2])] = -1;
  }
}

__global__ void k_count_pores(const int32_t* __restrict__ phase, long long N, unsigned long long* __restrict__ count) {
  unsigned long long c = 0;
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < N; v += (long long)gridDim.x * blockDim.x)
    c += phase[v] < 0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xffffffffu, c, o);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(count, c);
}

bool finite_all(const double* p, size_t n) {
  for (size_t t = 0; t < n; ++t)
    if (!std::isfinite(p[t])) return false;
  return true;
}

int sm_count() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return 0;
  return sms;
}

}  // namespace

int gen_error(int code, const std::string& m) { return gen_fail(code, m); }
}  // namespace elas

using namespace elas;

extern "C" {

const char* elas_generate_last_error(void) { return g_gen_err.c_str(); }

int elas_generate_workspace_bytes(int nx, int ny, int nz, int n_grains, int n_pores, size_t* bytes) {
  if (!bytes || nx < 1 || ny < 1 || nz < 1 || n_grains < 0 || n_pores < 0)
    return gen_fail(ELAS_ERR_INVALID_ARG, "elas_generate_workspace_bytes: bad arguments");
  *bytes = gen_layout(gen_grid(nx, ny, nz, n_grains), n_grains, n_pores).total;
  return ELAS_OK;
}

int elas_assign_grains(int nx, int ny, int nz, const double* seeds, const double* semi_axes, int n_grains,
                       int32_t* phase, void* workspace, size_t ws_bytes, void* cuda_stream) {
  if (nx < 1 || ny < 1 || nz < 1 || n_grains < 1 || !seeds || !phase)
    return gen_fail(ELAS_ERR_INVALID_ARG, "elas_assign_grains: bad dimensions, grain count or pointer");
  if ((long long)nx * ny * nz > (1LL << 31) - 1) return gen_fail(ELAS_ERR_INVALID_ARG, "elas_assign_grains: grid too large");
  const double L[3] = {(double)nx, (double)ny, (double)nz};
  for (int l = 0; l < n_grains; ++l)
    for (int d = 0; d < 3; ++d)
      if (!(seeds[3 * l + d] >= 0.0 && seeds[3 * l + d] < L[d]))
        return gen_fail(ELAS_ERR_INVALID_ARG, "elas_assign_grains: a seed lies outside [0, n) in some dimension");
  double rmax = 1.0;
  if (semi_axes) {
    rmax = 0.0;
    for (int t = 0; t < 2 * n_grains; ++t) {
      if (!(semi_axes[t] > 0.0) || !std::isfinite(semi_axes[t]))
        return gen_fail(ELAS_ERR_INVALID_ARG, "elas_assign_grains: semi-axes must be positive and finite");
      rmax = std::max(rmax, semi_axes[t]);
    }
  }
  GenGrid G = gen_grid(nx, ny, nz, n_grains);
  G.inv_rmax2 = 1.0 / (rmax * rmax);
  const GenLayout Ly = gen_layout(G, n_grains, 0);
  if (!workspace || ((uintptr_t)workspace % 256) != 0 || ws_bytes < Ly.total)
    return gen_fail(ELAS_ERR_WORKSPACE, "elas_assign_grains: workspace too small or not 256-byte aligned");
  // bin the seeds (counting sort by cell, grain order kept within a cell)
  const int cells = G.g[0] * G.g[1] * G.g[2];
  std::vector<int> start(cells + 1, 0), items(n_grains), cell_of(n_grains);
  for (int l = 0; l < n_grains; ++l) {
    int c[3];
    for (int d = 0; d < 3; ++d) c[d] = std::min(G.g[d] - 1, std::max(0, (int)std::floor(seeds[3 * l + d] / G.cs[d])));
    cell_of[l] = c[0] + G.g[0] * (c[1] + G.g[1] * c[2]);
    ++start[cell_of[l] + 1];
  }
  for (int c = 0; c < cells; ++c) start[c + 1] += start[c];
  std::vector<int> fill(start.begin(), start.end() - 1);
  for (int l = 0; l < n_grains; ++l) items[fill[cell_of[l]]++] = l;
  // in cell order: seeds, semi-axes, and for the FP32 screen the seeds as float pairs with the
  // weights (rmax / r)^2
  std::vector<double> sorted(3 * (size_t)n_grains), sorted_semi(semi_axes ? 2 * (size_t)n_grains : 0);
  std::vector<float4> fast(2 * (size_t)n_grains);
  double rmin = rmax;
  for (int t = 0; t < n_grains; ++t) {
    float hi[3], lo[3], w[2] = {1.f, 1.f};
    for (int d = 0; d < 3; ++d) {
      const double v = seeds[3 * (size_t)items[t] + d];
      sorted[3 * (size_t)t + d] = v;
      hi[d] = (float)v;
      lo[d] = (float)(v - (double)hi[d]);
    }
    for (int d = 0; semi_axes && d < 2; ++d) {
      const double r = semi_axes[2 * (size_t)items[t] + d];
      sorted_semi[2 * (size_t)t + d] = r;
      w[d] = (float)((rmax / r) * (rmax / r));
      rmin = std::min(rmin, r);
    }
    fast[2 * (size_t)t] = make_float4(hi[0], hi[1], hi[2], w[0]);
    fast[2 * (size_t)t + 1] = make_float4(lo[0], lo[1], lo[2], w[1]);
  }
  // the FP32 screen needs half-integers that are exact in float, distances (up to rmax / rmin squared
  // times the cell's) inside the float range and FP64 distances that neither overflow nor underflow
  const bool screen = rmax <= 1e6 * rmin && rmin > 1e-100 && rmax < 1e100 && std::max(nx, std::max(ny, nz)) <= (1 << 21);
  char* base = (char*)workspace;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  cudaError_t e = cudaMemcpyAsync(base + Ly.seeds, sorted.data(), sizeof(double) * sorted.size(), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess && semi_axes)
    e = cudaMemcpyAsync(base + Ly.semi, sorted_semi.data(), sizeof(double) * sorted_semi.size(), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(base + Ly.fast, fast.data(), sizeof(float4) * fast.size(), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(base + Ly.start, start.data(), sizeof(int) * start.size(), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(base + Ly.items, items.data(), sizeof(int) * items.size(), cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return gen_fail(ELAS_ERR_CUDA, std::string("elas_assign_grains: ") + cudaGetErrorString(e));
  const int sms = std::max(sm_count(), 1);
  const double* d_seeds = (const double*)(base + Ly.seeds);
  const double* d_semi = semi_axes ? (const double*)(base + Ly.semi) : nullptr;
  const int *d_start = (const int*)(base + Ly.start), *d_items = (const int*)(base + Ly.items);
  if (screen) {
    const long long tiles = (long long)((nx - 1) / kTile + 1) * ((ny - 1) / kTile + 1) * ((nz - 1) / kTile + 1);
    const int blocks = (int)std::min<long long>(tiles, (long long)sms * 32);
    auto kern = semi_axes ? k_assign<true> : k_assign<false>;
    kern<<<blocks, kGenThreads, 0, s>>>(nx, ny, nz, d_seeds, d_semi, (const float4*)(base + Ly.fast), n_grains, d_start,
                                        d_items, G, phase);
  } else {
    const long long N = (long long)nx * ny * nz;
    const int blocks = (int)std::min<long long>((N + kGenThreads - 1) / kGenThreads, (long long)sms * 32);
    auto kern = semi_axes ? k_assign_exact<true> : k_assign_exact<false>;
    kern<<<blocks, kGenThreads, 0, s>>>(nx, ny, nz, d_seeds, d_semi, n_grains, d_start, d_items, G, phase);
  }
  e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);  // the host tables above go out of scope
  if (e != cudaSuccess) return gen_fail(ELAS_ERR_CUDA, std::string("elas_assign_grains: ") + cudaGetErrorString(e));
  return ELAS_OK;
}

int elas_stamp_pores(int nx, int ny, int nz, const double* pores, int n_pores, int32_t* phase,
                     long long* n_pore_voxels, void* workspace, size_t ws_bytes, void* cuda_stream) {
  if (nx < 1 || ny < 1 || nz < 1 || n_pores < 0 || (n_pores > 0 && !pores) || !phase)
    return gen_fail(ELAS_ERR_INVALID_ARG, "elas_stamp_pores: bad dimensions, pore count or pointer");
  if ((long long)nx * ny * nz > (1LL << 31) - 1) return gen_fail(ELAS_ERR_INVALID_ARG, "elas_stamp_pores: grid too large");
  const double L[3] = {(double)nx, (double)ny, (double)nz};
  if (n_pores > 0 && !finite_all(pores, (size_t)kPoreDoubles * n_pores))
    return gen_fail(ELAS_ERR_INVALID_ARG, "elas_stamp_pores: non-finite pore parameter");
  for (int p = 0; p < n_pores; ++p) {
    const double* P = pores + kPoreDoubles * p;
    for (int d = 0; d < 3; ++d) {
      if (!(P[d] >= 0.0 && P[d] < L[d]))
        return gen_fail(ELAS_ERR_INVALID_ARG, "elas_stamp_pores: a pore centre lies outside the grid");
      // the minimum image sees a pore whole only when it is shorter than half the cell
      if (!(P[3 + d] > 0.0) || !(P[3 + d] < 0.5 * std::min(L[0], std::min(L[1], L[2]))))
        return gen_fail(ELAS_ERR_INVALID_ARG, "elas_stamp_pores: semi-axes must be positive and below half the cell");
    }
  }
  const GenLayout Ly = gen_layout(gen_grid(nx, ny, nz, 1), 0, n_pores);
  if (!workspace || ((uintptr_t)workspace % 256) != 0 || ws_bytes < Ly.total)
    return gen_fail(ELAS_ERR_WORKSPACE, "elas_stamp_pores: workspace too small or not 256-byte aligned");
  char* base = (char*)workspace;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  cudaError_t e = cudaSuccess;
  if (n_pores > 0)
    e = cudaMemcpyAsync(base + Ly.pores, pores, sizeof(double) * kPoreDoubles * n_pores, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(base + Ly.counter, 0, sizeof(unsigned long long) * 2, s);
  if (e == cudaSuccess && n_pores > 0) {
    // about 1,024 voxels of the largest pore's box per block
    double amax = 0.0;
    for (int p = 0; p < n_pores; ++p)
      for (int d = 0; d < 3; ++d) amax = std::max(amax, pores[kPoreDoubles * p + 3 + d]);
    const double box = std::pow(2.0 * std::ceil(amax) + 3.0, 3.0);
    const int split = (int)std::min(256.0, std::max(1.0, box / 1024.0));
    k_stamp<<<dim3(n_pores, split), kGenThreads, 0, s>>>(nx, ny, nz, (const double*)(base + Ly.pores), phase);
    e = cudaGetLastError();
  }
  const long long N = (long long)nx * ny * nz;
  if (e == cudaSuccess) {
    const int sms = std::max(sm_count(), 1);
    const long long blocks = std::min<long long>((N + kGenThreads - 1) / kGenThreads, (long long)sms * 8);
    k_count_pores<<<(int)blocks, kGenThreads, 0, s>>>(phase, N, (unsigned long long*)(base + Ly.counter));
    e = cudaGetLastError();
  }
  unsigned long long cnt = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&cnt, base + Ly.counter, sizeof cnt, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return gen_fail(ELAS_ERR_CUDA, std::string("elas_stamp_pores: ") + cudaGetErrorString(e));
  if (n_pore_voxels) *n_pore_voxels = (long long)cnt;
  return ELAS_OK;
}

}  // extern "C"
