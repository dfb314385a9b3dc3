// Maximum-stress extraction (ELAS3D-Xtal, arXiv 2602.07354, App. C): the von Mises field is
// smoothed by a normalised (masked) Gaussian convolution, smooth = G * (vm M) / G * M with M the
// solid indicator, on the periodic cell; the hotspots are the solid voxels that no competing
// 26-neighbour exceeds (every neighbour, or the solid ones only), and the stress concentration
// uses the largest of them.  The sums run over dz, dy, dx
// with the weight (w[dz] * w[dy]) * w[dx], every operation explicitly rounded, so the field is
// bitwise the same as a plain loop in that order; the maximum (and the lowest voxel id holding it)
// does not depend on the order in which blocks finish.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cstdlib>

#include "column_tile.h"

namespace elas {

namespace {

constexpr int kHotThreads = 512;

// Weights by class (|dz|, |dy|, |dx|), rounded as (w[dz] * w[dy]) * w[dx]; the sum of all weights in
// the order of the taps and its reciprocal.
struct Weights {
  double w[(kHotMaxRadius + 1) * (kHotMaxRadius + 1) * (kHotMaxRadius + 1)];
  double full, inv_full;
};

__device__ __forceinline__ int wrapn(int i, int n) {
  i %= n;
  return i < 0 ? i + n : i;
}

// One item = a tile of tx x ty voxel columns and zc layers; thread t owns column (t % tx, t / tx) and
// marches z.  Plane p adds its taps to the 2R + 1 outputs it reaches (dz = p - z rises with p, so
// every output meets its taps in the order dz, dy, dx); a pore's tap adds +0, which changes nothing.
//
// Bound: the FP64 pipe (1.66 operations per SM and clock).  The operations that the rounding order
// leaves are 27 sums a voxel (R = 1); a plain loop spent 4 per tap (two for the weight and its sum).
// Here a voxel's products with the 8 weight classes are formed once and shared through shared memory
// (9.6 a voxel with the tile's halo, instead of 27), the weight sum is the constant full sum unless
// the window holds a pore, and the division by that constant is a multiplication by its correctly
// rounded reciprocal and one residual correction (Markstein 1990: correctly rounded).  200^3, s = 0.4:
// 2.05 -> 0.84 ms, FP64 pipe 82% busy.
// For R >= 2 the classes outgrow shared memory: one product per tap and |dz|, shared by the outputs on
// either side.  The planes beside an item reach only some of its outputs; computing all of them made
// items of few layers (small grids) up to six times slower than a plain loop (the call on 24^3, s = 1.9:
// 281 us with the loop, 1,660, 201 now; 48^3, s = 0.8: 176, 250, 151).  200^3, s = 0.8, 1.2 and 1.9:
// 8.86, 22.3 and 46.2 ms with the loop, 4.47, 12.6 and 28.5 now.
template <int R, int NT>
__global__ void __launch_bounds__(NT, (R == 1 ? 2 : 1) * kHotThreads / NT)
    k_smooth(int nx, int ny, int nz, int tx, int ty, int zc, const int32_t* __restrict__ phase,
             const double* __restrict__ vm, const __grid_constant__ Weights W, double* __restrict__ smooth) {
  constexpr int D = 2 * R + 1, C = R + 1, NQ = R == 1 ? 8 : 1;
  constexpr int kPos = 3;  // staged positions per thread
  extern __shared__ __align__(16) unsigned char hot_smem[];
  const int t = threadIdx.x, wx = tx + 2 * R, wy = ty + 2 * R, np = wx * wy;
  double* const val = reinterpret_cast<double*>(hot_smem);            // [2][NQ][np]
  unsigned char* const sol = reinterpret_cast<unsigned char*>(val + 2 * NQ * np);  // [2][np]
  const int bx = (nx - 1) / tx + 1, by = (ny - 1) / ty + 1, bz = (nz - 1) / zc + 1;
  const long long plane = (long long)nx * ny;
  const int i = t % tx, j = t / tx;
  const bool own = j < ty;
  for (long long item = blockIdx.x; item < (long long)bx * by * bz; item += gridDim.x) {
    const int i0 = (int)(item % bx) * tx, j0 = (int)((item / bx) % by) * ty, z0 = (int)(item / ((long long)bx * by)) * zc;
    const int z1 = min(z0 + zc, nz);
    int off[kPos];
#pragma unroll
    for (int q = 0; q < kPos; ++q) {
      const int s = t + q * NT;
      off[q] = s < np ? wrapn(j0 - R + s / wx, ny) * nx + wrapn(i0 - R + s % wx, nx) : -1;
    }
    double pv[kPos];
    int pp[kPos];
    auto fetch = [&](int p) {
      const long long base = wrapn(p, nz) * plane;
#pragma unroll
      for (int q = 0; q < kPos; ++q)
        if (off[q] >= 0) {
          pv[q] = vm[base + off[q]];
          pp[q] = phase[base + off[q]];
        }
    };
    double acc[D];
    unsigned mask[D];  // solid taps of the planes met so far, oldest first (R = 1: 9 bits a plane)
#pragma unroll
    for (int d = 0; d < D; ++d) {
      acc[d] = 0.0;
      mask[d] = 0;
    }
    bool whole[D] = {};  // plane without a pore in the window
    const bool valid = own && i0 + i < nx && j0 + j < ny;
    fetch(z0 - R);
    for (int p = z0 - R; p < z1 + R; ++p) {
      const int b = (p - z0 + R) & 1;
      double* const v = val + b * NQ * np;
      unsigned char* const so = sol + b * np;
#pragma unroll
      for (int q = 0; q < kPos; ++q)
        if (off[q] >= 0) {
          const int s = t + q * NT;
          const bool solid = pp[q] >= 0;
          so[s] = solid;
          if constexpr (R == 1) {
#pragma unroll
            for (int c = 0; c < NQ; ++c) v[c * np + s] = solid ? __dmul_rn(W.w[c], pv[q]) : 0.0;
          } else {
            v[s] = solid ? pv[q] : 0.0;
          }
        }
      if (p + 1 < z1 + R) fetch(p + 1);
      __syncthreads();  // (the other buffer's readers have passed the last one)
      if (valid) {
        bool all = true;
        unsigned m = 0;
        if constexpr (R == 1) {
          // (the planes beside the item's layers reach only one of the three outputs)
          const bool up = p + 1 < z1, here = p >= z0 && p < z1, down = p > z0;
#pragma unroll
          for (int dy = 0; dy < 3; ++dy) {
            double far[3], near[3];
#pragma unroll
            for (int dx = 0; dx < 3; ++dx) {
              const int s = (j + dy) * wx + i + dx, c = (dy == 1 ? 0 : 2) + (dx == 1 ? 0 : 1);
              m |= (unsigned)so[s] << (3 * dy + dx);
              far[dx] = v[(4 + c) * np + s];
              near[dx] = v[c * np + s];
            }
            if (up) {  // output p + 1
#pragma unroll
              for (int dx = 0; dx < 3; ++dx) acc[0] = __dadd_rn(acc[0], far[dx]);
            }
            if (here) {  // output p
#pragma unroll
              for (int dx = 0; dx < 3; ++dx) acc[1] = __dadd_rn(acc[1], near[dx]);
            }
            if (down) {  // output p - 1: complete
#pragma unroll
              for (int dx = 0; dx < 3; ++dx) acc[2] = __dadd_rn(acc[2], far[dx]);
            }
          }
          all = m == 0x1ff;
        } else {
          // outputs p + cz and p - cz, as far as the item owns them (one cz after the other: an output meets
          // the plane's taps in one of the loops, in the order dy, dx)
#pragma unroll
          for (int cz = 0; cz <= R; ++cz) {
            const bool up = p + cz >= z0 && p + cz < z1, down = cz && p - cz >= z0 && p - cz < z1;
            if (!up && !down) continue;
            double a = acc[R - cz], b = acc[R + cz];
#pragma unroll
            for (int dy = 0; dy < D; ++dy)
#pragma unroll
              for (int dx = 0; dx < D; ++dx) {
                const int cy = dy < R ? R - dy : dy - R, cx = dx < R ? R - dx : dx - R;
                const double q = __dmul_rn(W.w[(cz * C + cy) * C + cx], v[(j + dy) * wx + i + dx]);
                if (up) a = __dadd_rn(a, q);
                if (down) b = __dadd_rn(b, q);
              }
            acc[R - cz] = a;
            if (cz) acc[R + cz] = b;
          }
          for (int dy = 0; dy < D; ++dy)
#pragma unroll
            for (int dx = 0; dx < D; ++dx) all = all && so[(j + dy) * wx + i + dx];
        }
#pragma unroll
        for (int d = 0; d < D - 1; ++d) {
          whole[d] = whole[d + 1];
          mask[d] = mask[d + 1];
        }
        whole[D - 1] = all;
        mask[D - 1] = m;
        const int z = p - R;
        if (z >= z0) {
          bool full = true;
#pragma unroll
          for (int d = 0; d < D; ++d) full = full && whole[d];
          const double num = acc[D - 1];
          const long long n = z * plane + (long long)(j0 + j) * nx + i0 + i;
          const int e = (__double2hiint(num) >> 20) & 0x7ff;  // exponent field: 2^-930 .. 2^930 passes
          if (full && e > 93 && e < 1953) {
            const double q = __dmul_rn(num, W.inv_full);
            smooth[n] = __fma_rn(__fma_rn(-q, W.full, num), W.inv_full, q);
          } else {
            double den = full ? W.full : 0.0;
            if (!full) {
              if constexpr (R == 1) {
#pragma unroll
                for (int d = 0; d < 27; ++d) {
                  const int dz = d / 9, dy = (d / 3) % 3, dx = d % 3;
                  if ((mask[dz] >> (d % 9)) & 1)
                    den = __dadd_rn(den, W.w[(dz == 1 ? 0 : 4) + (dy == 1 ? 0 : 2) + (dx == 1 ? 0 : 1)]);
                }
              } else {
                for (int dz = -R; dz <= R; ++dz)
                  for (int dy = -R; dy <= R; ++dy)
                    for (int dx = -R; dx <= R; ++dx)
                      if (phase[wrapn(z + dz, nz) * plane + (long long)wrapn(j0 + j + dy, ny) * nx + wrapn(i0 + i + dx, nx)] >= 0)
                        den = __dadd_rn(den, W.w[(abs(dz) * C + abs(dy)) * C + abs(dx)]);
              }
            }
            smooth[n] = den > 0.0 ? __ddiv_rn(num, den) : 0.0;
          }
        }
#pragma unroll
        for (int d = D - 1; d > 0; --d) acc[d] = acc[d - 1];
        acc[0] = 0.0;
      }
    }
    __syncthreads();  // the next item stages into the buffers read last
  }
}

// Order-preserving integer of a double (equal zeros); NaN, which exceeds nothing, below all others.
__device__ __forceinline__ long long order_key(double x) {
  const long long b = __double_as_longlong(x);
  if ((b & LLONG_MAX) > 0x7ff0000000000000ll) return LLONG_MIN;
  return b >= 0 ? b : (b == LLONG_MIN ? 0 : b ^ LLONG_MAX);
}

__device__ __forceinline__ void better(unsigned long long& bits, unsigned long long& vox, unsigned long long b,
                                       unsigned long long v) {
  if (b > bits || (b == bits && v < vox)) {
    bits = b;
    vox = v;
  }
}

// The largest hotspot value (as its bits, compared unsigned) and the lowest voxel holding it, in one
// pass: thread t marches z through its column with the 3 x 3 maxima of three planes, compared as
// order-preserving integers (26 FP64 comparisons a voxel and pass would be bound by the FP64 pipe:
// 200^3: two passes 0.84 ms, this one 0.10).  Each block leaves its best in a slot; the last one to finish reduces them.
__global__ void __launch_bounds__(kHotThreads)
    k_hotspot(int nx, int ny, int nz, int tx, int ty, int zc, const int32_t* __restrict__ phase,
              const double* __restrict__ smooth, bool solid_only, unsigned long long* __restrict__ best,
              unsigned int* __restrict__ ctr, unsigned long long* __restrict__ slots) {
  constexpr int kPos = 2;
  extern __shared__ __align__(16) unsigned char hot_smem[];
  __shared__ unsigned long long rb[kHotThreads / 32], rv[kHotThreads / 32];
  __shared__ int last;
  const int t = threadIdx.x, wx = tx + 2, np = wx * (ty + 2);
  long long* const key = reinterpret_cast<long long*>(hot_smem);                      // [2][np]
  unsigned char* const sol = reinterpret_cast<unsigned char*>(key + 2 * np);           // [2][np]
  const int bx = (nx - 1) / tx + 1, by = (ny - 1) / ty + 1, bz = (nz - 1) / zc + 1;
  const long long plane = (long long)nx * ny;
  const int i = t % tx, j = t / tx;
  unsigned long long bits = 0ull, vox = ~0ull;
  for (long long item = blockIdx.x; item < (long long)bx * by * bz; item += gridDim.x) {
    const int i0 = (int)(item % bx) * tx, j0 = (int)((item / bx) % by) * ty, z0 = (int)(item / ((long long)bx * by)) * zc;
    const int z1 = min(z0 + zc, nz);
    int off[kPos];
#pragma unroll
    for (int q = 0; q < kPos; ++q) {
      const int s = t + q * kHotThreads;
      off[q] = s < np ? wrapn(j0 - 1 + s / wx, ny) * nx + wrapn(i0 - 1 + s % wx, nx) : -1;
    }
    double pv[kPos];
    int pp[kPos];
    auto fetch = [&](int p) {
      const long long base = wrapn(p, nz) * plane;
#pragma unroll
      for (int q = 0; q < kPos; ++q)
        if (off[q] >= 0) {
          pv[q] = smooth[base + off[q]];
          pp[q] = phase[base + off[q]];
        }
    };
    const bool valid = j < ty && i0 + i < nx && j0 + j < ny;
    long long m0 = LLONG_MIN, m1 = LLONG_MIN, self1 = 0;  // plane maxima of p - 2, p - 1; own key of p - 1
    bool solid1 = false;
    fetch(z0 - 1);
    for (int p = z0 - 1; p <= z1; ++p) {
      const int b = (p - z0 + 1) & 1;
      long long* const k = key + b * np;
      unsigned char* const so = sol + b * np;
#pragma unroll
      for (int q = 0; q < kPos; ++q)
        if (off[q] >= 0) {
          const int s = t + q * kHotThreads;
          so[s] = pp[q] >= 0;
          k[s] = solid_only && pp[q] < 0 ? LLONG_MIN : order_key(pv[q]);
        }
      if (p < z1) fetch(p + 1);
      __syncthreads();
      if (valid) {
        const int s = j * wx + i;
        long long m = k[s];
#pragma unroll
        for (int q = 1; q < 9; ++q) m = max(m, k[s + (q / 3) * wx + q % 3]);
        if (p > z0 && solid1) {
          const long long self = self1 == LLONG_MIN ? LLONG_MAX : self1;  // no neighbour exceeds a NaN
          if (self >= max(m0, max(m1, m))) {
            const long long n = (p - 1) * plane + (long long)(j0 + j) * nx + i0 + i;
            better(bits, vox, (unsigned long long)__double_as_longlong(smooth[n]), (unsigned long long)n);
          }
        }
        m0 = m1;
        m1 = m;
        self1 = k[s + wx + 1];
        solid1 = so[s + wx + 1];
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long b = __shfl_down_sync(0xffffffffu, bits, o), v = __shfl_down_sync(0xffffffffu, vox, o);
    better(bits, vox, b, v);
  }
  if ((t & 31) == 0) {
    rb[t / 32] = bits;
    rv[t / 32] = vox;
  }
  __syncthreads();
  if (t == 0) {
    for (int w = 1; w < kHotThreads / 32; ++w) better(bits, vox, rb[w], rv[w]);
    slots[2 * blockIdx.x] = bits;
    slots[2 * blockIdx.x + 1] = vox;
    __threadfence();
    last = atomicAdd(ctr, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  bits = 0ull;
  vox = ~0ull;
  for (int q = t; q < (int)gridDim.x; q += kHotThreads) better(bits, vox, __ldcg(slots + 2 * q), __ldcg(slots + 2 * q + 1));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long b = __shfl_down_sync(0xffffffffu, bits, o), v = __shfl_down_sync(0xffffffffu, vox, o);
    better(bits, vox, b, v);
  }
  __syncthreads();
  if ((t & 31) == 0) {
    rb[t / 32] = bits;
    rv[t / 32] = vox;
  }
  __syncthreads();
  if (t == 0) {
    for (int w = 1; w < kHotThreads / 32; ++w) better(bits, vox, rb[w], rv[w]);
    best[0] = bits;
    best[1] = vox;
  }
}

// Block size, tile and layers of the smoothing: the busiest SM's FP64 operations (an output layer's, a
// staged position's and, for R >= 2, those that an item's ends add), with a plane's barrier and load
// counted as 3,300 (2,000 clocks).  Fewer threads than `few` on an SM wait for their own sums instead of
// for the pipe.
template <int R>
ColumnTile smooth_tile(const Geo& g, int sm_count) {
  constexpr int D = 2 * R + 1;
  constexpr double layer = R == 1 ? 30 : D * D * (3 * R + 2), pos = R == 1 ? 8 : 0, ends = R == 1 ? 0 : D * D * R;
  ColumnTile best{};
  double cost0 = 1e300;
  for (int threads = kHotThreads; threads >= 128; threads /= 2) {
    ColumnTile h = column_tile(g, threads, 2 * R, 2 * R, 1.0, sm_count, R == 1 ? std::min(704, 3 * threads) : 3 * threads);
    const int tiles = h.items / ((g.nz - 1) / h.zc + 1), last = h.zc;
    for (int zc = R == 1 ? last : 1; zc <= last; zc = next_chunk(g.nz, zc)) {
      const long long items = (long long)tiles * ((g.nz - 1) / zc + 1), m = (items + sm_count - 1) / sm_count;
      if (items > (1 << 30)) continue;
      const double few = R == 1 ? 0 : 224;
      const double cost = std::max((double)m * threads, few) * (layer * zc + ends) +
                          m * (zc + 2 * R) * (pos * (h.tx + 2 * R) * (h.ty + 2 * R) + 3300.0);
      if (cost < cost0) {
        cost0 = cost;
        best = h;
        best.threads = threads;
        best.zc = zc;
        best.items = (int)items;
      }
    }
    // R = 1 from 64^3 on: smaller blocks give nothing and looking at them 3 us of a call of 94
    if (R == 1 && last >= 4) break;
  }
  return best;
}

template <int R, int NT>
cudaError_t launch_smooth_t(const Geo& g, const ColumnTile& h, const int32_t* phase, const double* vm, const Weights& W,
                            double* smooth, cudaStream_t s) {
  constexpr int NQ = R == 1 ? 8 : 1, most = 2 * (R == 1 ? std::min(704, 3 * NT) : 3 * NT) * (8 * NQ + 1);
  const size_t smem = (size_t)(h.tx + 2 * R) * (h.ty + 2 * R) * 2 * (NQ * sizeof(double) + 1);
  cudaError_t e = cudaFuncSetAttribute(k_smooth<R, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  if (e != cudaSuccess) return e;
  k_smooth<R, NT><<<h.items, NT, smem, s>>>(g.nx, g.ny, g.nz, h.tx, h.ty, h.zc, phase, vm, W, smooth);
  return cudaGetLastError();
}

template <int R>
cudaError_t launch_smooth(const Geo& g, const int32_t* phase, const double* vm, const Weights& W, double* smooth,
                          int sm_count, cudaStream_t s) {
  const ColumnTile h = smooth_tile<R>(g, sm_count);
  return h.threads == 128   ? launch_smooth_t<R, 128>(g, h, phase, vm, W, smooth, s)
         : h.threads == 256 ? launch_smooth_t<R, 256>(g, h, phase, vm, W, smooth, s)
                            : launch_smooth_t<R, kHotThreads>(g, h, phase, vm, W, smooth, s);
}

}  // namespace

cudaError_t launch_hotspot(const Geo& g, const int32_t* phase, const double* vm, double s_kernel, bool solid_only,
                           double* smooth, unsigned long long* best2, int sm_count, cudaStream_t s) {
  const int r = hot_radius(s_kernel);
  double w[2 * kHotMaxRadius + 1];
  hot_weights(s_kernel, r, w);
  Weights W{};
  for (int cz = 0; cz <= r; ++cz)
    for (int cy = 0; cy <= r; ++cy)
      for (int cx = 0; cx <= r; ++cx) W.w[(cz * (r + 1) + cy) * (r + 1) + cx] = (w[r + cz] * w[r + cy]) * w[r + cx];
  W.full = 0.0;
  for (int dz = -r; dz <= r; ++dz)
    for (int dy = -r; dy <= r; ++dy)
      for (int dx = -r; dx <= r; ++dx) W.full += W.w[(std::abs(dz) * (r + 1) + std::abs(dy)) * (r + 1) + std::abs(dx)];
  W.inv_full = 1.0 / W.full;
  cudaError_t e = r == 1   ? launch_smooth<1>(g, phase, vm, W, smooth, sm_count, s)
                  : r == 2 ? launch_smooth<2>(g, phase, vm, W, smooth, sm_count, s)
                  : r == 3 ? launch_smooth<3>(g, phase, vm, W, smooth, sm_count, s)
                           : launch_smooth<4>(g, phase, vm, W, smooth, sm_count, s);
  // best2: the result (2 values), the arrival counter, and the blocks' slots
  unsigned int* ctr = reinterpret_cast<unsigned int*>(best2 + 2);
  if (e == cudaSuccess) e = cudaMemsetAsync(ctr, 0, sizeof(unsigned int), s);
  if (e != cudaSuccess) return e;
  const ColumnTile h = column_tile(g, kHotThreads, 2, 2, 1, sm_count, 2 * kHotThreads);
  const size_t smem = (size_t)(h.tx + 2) * (h.ty + 2) * 2 * (sizeof(long long) + 1);
  k_hotspot<<<std::min(h.items, kMaxParts), kHotThreads, smem, s>>>(
      g.nx, g.ny, g.nz, h.tx, h.ty, h.zc, phase, smooth, solid_only, best2, ctr, best2 + 8);
  return cudaGetLastError();
}

}  // namespace elas
