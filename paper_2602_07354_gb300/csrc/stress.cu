// Voxel stress, von Mises and macroscopic stress (stress_OpenMP / stress_fullfield_OpenMP of
// ELAS3D-Xtal, arXiv 2602.07354, Table 1): strain at the voxel centroid (the exact voxel average of
// the trilinear field), sigma = C eps, and the mean stress over all voxels.
#include <cuda_runtime.h>

#include <algorithm>

#include "column_tile.h"

namespace elas {

namespace {

constexpr int kStressThreads = 256;
constexpr int kStressPos = 2;  // staged node pairs per thread

__device__ __forceinline__ int wrap1(int i, int n) {
  i %= n;
  return i < 0 ? i + n : i;
}

// Sums of six values over the block, thread 0's result (a fixed order): the first step pairs two
// values in the two half-warps, so a warp spends 15 FP64 additions instead of 30.
__device__ void block_sum6(const double (&a)[6], double (&out)[6], double* red) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  double v[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const double mine = lane < 16 ? a[2 * q] : a[2 * q + 1], other = lane < 16 ? a[2 * q + 1] : a[2 * q];
    v[q] = mine + __shfl_xor_sync(0xffffffffu, other, 16);
  }
#pragma unroll
  for (int o = 8; o > 0; o >>= 1)
#pragma unroll
    for (int q = 0; q < 3; ++q) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
  __syncthreads();
  if ((lane & 15) == 0) {
#pragma unroll
    for (int q = 0; q < 3; ++q) red[6 * wid + 2 * q + (lane >> 4)] = v[q];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      out[q] = 0.0;
      for (int w = 0; w < kStressThreads / 32; ++w) out[q] += red[6 * w + q];
    }
  }
}

struct Strain {
  double e[6];  // E11, E22, E33, 2 E23, 2 E13, 2 E12
};

// One item = a tile of tx x ty voxel columns and zc layers; thread t owns column (t % tx, t / tx) and
// marches z.  A node plane is staged as sums and differences of x neighbours, so that a face's four
// corners give their sum and their two differences with three additions a component, and a voxel's
// centroid gradient (d w_c / d x_d = sum_a s_d(a) w_ac / 4) takes its lower face's values from the
// voxel below.
//
// Bound: the FP64 pipe (1.66 operations per SM and clock): 24 multiply-adds a component in the
// gradient made 150 operations a voxel with the 36 of C eps, von Mises and the mean; with shared
// faces they are 96 (200^3, the call: 2.03 -> 1.52 ms, pipe 86% busy before and after).
__global__ void __launch_bounds__(kStressThreads, 2)
    k_stress(int nx, int ny, int nz, int tx, int ty, int zc, long long N, const int32_t* __restrict__ phase,
             const double* __restrict__ cfull, const __grid_constant__ Strain E, const double* __restrict__ w,
             double* __restrict__ stress, double* __restrict__ vm, double* parts, unsigned int* ctr, double* macro_out) {
  extern __shared__ __align__(16) double st_smem[];  // [2][3 components][sum, difference][np]
  __shared__ double red[6 * kStressThreads / 32];
  __shared__ int last;
  const int t = threadIdx.x, np = tx * (ty + 1);
  const int bx = (nx - 1) / tx + 1, by = (ny - 1) / ty + 1, bz = (nz - 1) / zc + 1;
  const long long plane = (long long)nx * ny;
  const int i = t % tx, j = t / tx;
  double acc[6] = {0, 0, 0, 0, 0, 0};
  for (long long item = blockIdx.x; item < (long long)bx * by * bz; item += gridDim.x) {
    const int i0 = (int)(item % bx) * tx, j0 = (int)((item / bx) % by) * ty, z0 = (int)(item / ((long long)bx * by)) * zc;
    const int z1 = min(z0 + zc, nz);
    const bool valid = j < ty && i0 + i < nx && j0 + j < ny;
    int o0[kStressPos], o1[kStressPos];
#pragma unroll
    for (int q = 0; q < kStressPos; ++q) {
      const int s = t + q * kStressThreads;
      const int row = wrap1(j0 + s / tx, ny) * nx, x = i0 + s % tx;
      o0[q] = s < np ? row + wrap1(x, nx) : -1;
      o1[q] = row + wrap1(x + 1, nx);
    }
    double a[kStressPos][3], b[kStressPos][3];
    auto fetch = [&](int p) {
      const double* wp = w + (p < nz ? p : 0) * plane;
#pragma unroll
      for (int q = 0; q < kStressPos; ++q)
        if (o0[q] >= 0) {
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            a[q][c] = wp[c * N + o0[q]];
            b[q][c] = wp[c * N + o1[q]];
          }
        }
    };
    // the lower face: x difference of 0, y difference of 1, sum of 2, dy0 + dx1, dy2 - s1, dx2 - s0
    double lo[6];
    fetch(z0);
    for (int p = z0; p <= z1; ++p) {
      double* const f = st_smem + ((p - z0) & 1) * 6 * np;
#pragma unroll
      for (int q = 0; q < kStressPos; ++q)
        if (o0[q] >= 0) {
          const int s = t + q * kStressThreads;
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            f[2 * c * np + s] = a[q][c] + b[q][c];
            f[(2 * c + 1) * np + s] = b[q][c] - a[q][c];
          }
        }
      const long long n = (p - 1) * plane + (long long)(j0 + j) * nx + i0 + i;
      int ph = -1;
      if (valid && p > z0) ph = phase[n];
      if (p < z1) fetch(p + 1);
      __syncthreads();  // (the other buffer's readers have passed the last one)
      if (valid) {
        double S[3], Dx[3], Dy[3];
        const int s = t;  // = j tx + i
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const double s0 = f[2 * c * np + s], s1 = f[2 * c * np + s + tx];
          const double d0 = f[(2 * c + 1) * np + s], d1 = f[(2 * c + 1) * np + s + tx];
          S[c] = s0 + s1;
          Dy[c] = s1 - s0;
          Dx[c] = d0 + d1;
        }
        const double q5 = Dy[0] + Dx[1];
        if (p > z0) {
          double s6[6] = {0, 0, 0, 0, 0, 0};
          if (ph >= 0) {
            const double g[6] = {lo[0] + Dx[0], lo[1] + Dy[1], S[2] - lo[2], lo[4] + (Dy[2] + S[1]),
                                 lo[5] + (Dx[2] + S[0]), lo[3] + q5};
            double ev[6];
#pragma unroll
            for (int r = 0; r < 6; ++r) ev[r] = fma(0.25, g[r], E.e[r]);
            const double* C = cfull + (long long)ph * kSymStride;
#pragma unroll
            for (int r = 0; r < 6; ++r) {
              double v = C[pk(r, 0)] * ev[0];
#pragma unroll
              for (int c = 1; c < 6; ++c) v = fma(C[pk(r, c)], ev[c], v);
              s6[r] = v;
            }
          }
          if (stress) {
#pragma unroll
            for (int r = 0; r < 6; ++r) stress[r * N + n] = s6[r];
          }
          if (vm) {
            double m = 0.0;
            if (ph >= 0) {
              const double d1 = s6[0] - s6[1], d2 = s6[1] - s6[2], d3 = s6[2] - s6[0];
              m = sqrt(0.5 * (d1 * d1 + d2 * d2 + d3 * d3) + 3.0 * (s6[3] * s6[3] + s6[4] * s6[4] + s6[5] * s6[5]));
            }
            vm[n] = m;
          }
          if (macro_out) {
#pragma unroll
            for (int r = 0; r < 6; ++r) acc[r] += s6[r];
          }
        }
        lo[0] = Dx[0];
        lo[1] = Dy[1];
        lo[2] = S[2];
        lo[3] = q5;
        lo[4] = Dy[2] - S[1];
        lo[5] = Dx[2] - S[0];
      }
    }
    __syncthreads();  // the next item stages into the buffers read last
  }
  if (!macro_out) return;
  double sums[6];
  block_sum6(acc, sums, red);
  if (t == 0) {
    for (int r = 0; r < 6; ++r) parts[r * kMaxParts + blockIdx.x] = sums[r];
    __threadfence();
    last = atomicAdd(ctr, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  double tot[6] = {0, 0, 0, 0, 0, 0};
  for (int q = t; q < (int)gridDim.x; q += kStressThreads)
    for (int r = 0; r < 6; ++r) tot[r] += __ldcg(parts + r * kMaxParts + q);
  block_sum6(tot, sums, red);
  if (t == 0) {
    for (int r = 0; r < 6; ++r) macro_out[r] = sums[r] / (double)N;
    *ctr = 0u;
  }
}

}  // namespace

cudaError_t launch_stress(const Geo& g, const int32_t* phase, const double* cfull, const double* E6,
                          const double* w, double* stress, double* vm, double* parts, unsigned int* ctr,
                          double* macro_out, int sm_count, cudaStream_t s) {
  // one partial-sum slot per block; beyond kMaxParts items the blocks take several
  const ColumnTile h = column_tile(g, kStressThreads, 0, 1, 0.25, sm_count, kStressPos * kStressThreads, kMaxParts);
  const size_t smem = sizeof(double) * 2 * 6 * h.tx * (h.ty + 1);
  Strain e;
  for (int q = 0; q < 6; ++q) e.e[q] = q < 3 ? E6[q] : 2.0 * E6[q];
  k_stress<<<std::min(h.items, kMaxParts), kStressThreads, smem, s>>>(g.nx, g.ny, g.nz, h.tx, h.ty, h.zc, g.N, phase, cfull,
                                                                      e, w, stress, vm, parts, ctr, macro_out);
  return cudaGetLastError();
}

}  // namespace elas
