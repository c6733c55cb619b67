// FP32 inverse of the scaled Poisson matrix of a small planar mesh, computed on the device when the
// handle is created and applied by the AMG solvers as their preconditioner (AmgDenseT of level 0):
// the CG then needs two or three iterations of three grid-wide phases instead of ten of four to
// six.  4,225 nodes: 71 MB that stay in L2; a solve of 1.3 iterations takes 65 us over the whole GPU
// (199 us with the V-cycle on one cluster).
//
// In-place block Gauss-Jordan elimination without pivoting (the matrix is symmetric positive
// definite, so every pivot block is): with P = A_kk^-1, one step takes
//   A_kk <- P,   A_kj <- P A_kj,   A_ik <- -A_ik P,   A_ij <- A_ij - A_ik P A_kj.
// Two launches per block step: the pivot row's products (every thread block inverts the 64 x 64
// pivot itself, which is cheaper than a third launch) and the rank-64 update, 64 x 64 tiles of 4 x 4
// values per thread.  The result is symmetrised, as CG needs.
#include <cuda_runtime.h>

#include "avip_internal.h"

namespace avip {
namespace {
constexpr int kB = 64, kThreads = 256;

__global__ void dense_scatter_kernel(SellView A, int np, float* __restrict__ M) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= np) return;
  if (i >= A.N) {  // padding: an identity block
    M[(size_t)i * np + i] = 1.f;
    return;
  }
  const int e0 = A.sl_ptr[i / kSlice] + i % kSlice, rl = A.rlen[i];
  for (int k = 0; k < rl; ++k) M[(size_t)i * np + A.col[e0 + k * kSlice]] = (float)A.aval[e0 + k * kSlice];
}

// A 64 x 64 tile between global memory (row stride ld) and shared memory.
__device__ __forceinline__ void load_tile(float (*s)[kB + 4], const float* g, int ld) {
  for (int t = threadIdx.x; t < kB * kB / 4; t += kThreads) {
    const int r = t / (kB / 4), c = t % (kB / 4) * 4;
    *reinterpret_cast<float4*>(&s[r][c]) = *reinterpret_cast<const float4*>(g + (size_t)r * ld + c);
  }
}

// acc = X Y for this thread's 4 x 4 values (rows 4 ty .., columns 4 tx ..), X and Y in shared memory.
__device__ __forceinline__ void tile_product(float (&acc)[4][4], const float (*X)[kB + 4], const float (*Y)[kB + 4]) {
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[r][c] = 0.f;
#pragma unroll 4
  for (int k = 0; k < kB; k += 4) {
    float4 x[4], y[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) x[r] = *reinterpret_cast<const float4*>(&X[4 * ty + r][k]);
#pragma unroll
    for (int q = 0; q < 4; ++q) y[q] = *reinterpret_cast<const float4*>(&Y[k + q][4 * tx]);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float xv[4] = {x[r].x, x[r].y, x[r].z, x[r].w};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        acc[r][0] = fmaf(xv[q], y[q].x, acc[r][0]);
        acc[r][1] = fmaf(xv[q], y[q].y, acc[r][1]);
        acc[r][2] = fmaf(xv[q], y[q].z, acc[r][2]);
        acc[r][3] = fmaf(xv[q], y[q].w, acc[r][3]);
      }
    }
  }
}
__device__ __forceinline__ void store_tile(float* g, int ld, const float (&v)[4][4]) {
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
  for (int r = 0; r < 4; ++r)
    *reinterpret_cast<float4*>(g + (size_t)(4 * ty + r) * ld + 4 * tx) = make_float4(v[r][0], v[r][1], v[r][2], v[r][3]);
}

// Thread block j: P = A_kk^-1, R_j = P A_kj (R_k = P) and the copy C_j = A_jk (j != k).
//
// The pivot tile is inverted in registers, 16 columns of one row per thread (four neighbouring lanes
// hold a row): a step takes the pivot row from shared memory, two rows in turn so that one barrier per
// step suffices, and the thread's element of the pivot column from its quad by a shuffle.  Held in
// shared memory, with two barriers and 48 conflicting accesses per thread and step, the inversion took
// 77 us a launch.
__global__ void __launch_bounds__(kThreads) dense_pivot_kernel(const float* __restrict__ M, int np, int k,
                                                               float* __restrict__ R, float* __restrict__ Cc) {
  __shared__ float P[kB][kB + 4], Y[kB][kB + 4];
  __shared__ __align__(16) float pivot_row[2][kB];
  const int j = blockIdx.x;
  if (j != k) load_tile(Y, M + (size_t)k * kB * np + j * kB, np);
  const int r = threadIdx.x >> 2, q = threadIdx.x & 3, c0 = 16 * q;
  float v[16];
  const float4* src = reinterpret_cast<const float4*>(M + ((size_t)k * kB + r) * np + k * kB + c0);
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const float4 t = src[c];
    v[4 * c] = t.x, v[4 * c + 1] = t.y, v[4 * c + 2] = t.z, v[4 * c + 3] = t.w;
  }
#pragma unroll 1
  for (int pq = 0; pq < kB / 16; ++pq) {  // the pivot's quarter of the columns
#pragma unroll
    for (int pc = 0; pc < 16; ++pc) {
      const int p = 16 * pq + pc;
      float* row = pivot_row[pc & 1];
      if (r == p) {
#pragma unroll
        for (int c = 0; c < 4; ++c)
          *reinterpret_cast<float4*>(row + c0 + 4 * c) = make_float4(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
      }
      __syncthreads();
      const float piv = 1.f / row[p], f = __shfl_sync(0xffffffffu, v[pc], pq, 4) * piv;
#pragma unroll
      for (int c = 0; c < 16; ++c) {
        const bool pivot_column = q == pq && c == pc;
        if (r == p)
          v[c] = pivot_column ? piv : v[c] * piv;
        else
          v[c] = pivot_column ? -f : fmaf(-f, row[c0 + c], v[c]);
      }
    }
  }
  if (j == k) {
    float4* dst = reinterpret_cast<float4*>(R + (size_t)r * np + k * kB + c0);
#pragma unroll
    for (int c = 0; c < 4; ++c) dst[c] = make_float4(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
    return;
  }
#pragma unroll
  for (int c = 0; c < 4; ++c)
    *reinterpret_cast<float4*>(&P[r][c0 + 4 * c]) = make_float4(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
  __syncthreads();
  float acc[4][4];
  tile_product(acc, P, Y);
  store_tile(R + j * kB, np, acc);
  for (int t = threadIdx.x; t < kB * kB / 4; t += kThreads) {
    const int rr = t / (kB / 4), c = t % (kB / 4) * 4;
    *reinterpret_cast<float4*>(Cc + ((size_t)j * kB + rr) * kB + c) =
        *reinterpret_cast<const float4*>(M + ((size_t)j * kB + rr) * np + k * kB + c);
  }
}

// Tile (i, j) of the rank-64 update.
__global__ void __launch_bounds__(kThreads) dense_update_kernel(float* __restrict__ M, int np, int k,
                                                                const float* __restrict__ R,
                                                                const float* __restrict__ Cc) {
  __shared__ float X[kB][kB + 4], Y[kB][kB + 4];
  const int i = blockIdx.y, j = blockIdx.x;
  float* m = M + (size_t)i * kB * np + j * kB;
  load_tile(Y, R + j * kB, np);
  if (i == k) {  // the pivot row
    __syncthreads();
    for (int t = threadIdx.x; t < kB * kB / 4; t += kThreads) {
      const int r = t / (kB / 4), c = t % (kB / 4) * 4;
      *reinterpret_cast<float4*>(m + (size_t)r * np + c) = *reinterpret_cast<const float4*>(&Y[r][c]);
    }
    return;
  }
  load_tile(X, Cc + (size_t)i * kB * kB, kB);
  __syncthreads();
  float acc[4][4];
  tile_product(acc, X, Y);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const float4 old = j == k ? make_float4(0.f, 0.f, 0.f, 0.f)
                              : *reinterpret_cast<const float4*>(m + (size_t)(4 * ty + r) * np + 4 * tx);
    acc[r][0] = old.x - acc[r][0];
    acc[r][1] = old.y - acc[r][1];
    acc[r][2] = old.z - acc[r][2];
    acc[r][3] = old.w - acc[r][3];
  }
  store_tile(m, np, acc);
}

// M <- (M + M^T) / 2, tiles (i, j) and (j, i), i <= j.
__global__ void __launch_bounds__(kThreads) dense_symmetrise_kernel(float* __restrict__ M, int np) {
  __shared__ float X[kB][kB + 4], Y[kB][kB + 4];
  const int i = blockIdx.y, j = blockIdx.x;
  if (i > j) return;
  float *a = M + (size_t)i * kB * np + j * kB, *b = M + (size_t)j * kB * np + i * kB;
  load_tile(X, a, np);
  load_tile(Y, b, np);
  __syncthreads();
  for (int t = threadIdx.x; t < kB * kB; t += kThreads) {
    const int r = t / kB, c = t % kB;
    a[(size_t)r * np + c] = 0.5f * (X[r][c] + Y[c][r]);
    if (i != j) b[(size_t)r * np + c] = 0.5f * (Y[r][c] + X[c][r]);
  }
}
// Flags M when the largest row sum of |A M - I|, which bounds the spectral radius of A M - I, exceeds
// 1/2 in a row i (one thread block each; sums in FP64).
__global__ void __launch_bounds__(kThreads) dense_defect_kernel(SellView A, int np, const float* __restrict__ M,
                                                                int* __restrict__ bad) {
  __shared__ double part[kThreads / 32];
  const int i = blockIdx.x;
  const int e0 = A.sl_ptr[i / kSlice] + i % kSlice, rl = A.rlen[i];
  double sum = 0.0;
  for (int j = threadIdx.x; j < A.N; j += kThreads) {
    double d = i == j ? -1.0 : 0.0;
    for (int k = 0; k < rl; ++k) d = fma(A.aval[e0 + k * kSlice], (double)M[(size_t)A.col[e0 + k * kSlice] * np + j], d);
    sum += fabs(d);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (threadIdx.x % 32 == 0) part[threadIdx.x / 32] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kThreads / 32; ++w) sum += part[w];
    if (!(sum <= 0.5)) *bad = 1;  // (also for NaN)
  }
}
}  // namespace

// Rows of the padded matrix of N nodes.
int dense_inverse_rows(int N) { return (N + kB - 1) / kB * kB; }
// Floats of scratch: the pivot row and the pivot column.
size_t dense_inverse_scratch(int N) { return (size_t)2 * kB * dense_inverse_rows(N); }

// M (dense_inverse_rows squared, zeroed) becomes the inverse of A; *bad (zeroed) is set when FP32
// does not suffice: a matrix whose condition comes near 1e7 (cells of aspect 50 and more between
// electrodes at the long ends).  A spectral radius of A M - I of at most 1/2 keeps M positive
// definite and the CG's iterations few (condition of A M at most 3); ordinary meshes have 1e-6 to
// 1e-3.  With its memory it adds 8.3 ms to creating a handle of 4,608 nodes (4,225: 6.9, 1,353: 1.2).
cudaError_t launch_dense_inverse(const SellView& A, float* M, float* scratch, int* bad, cudaStream_t st) {
  const int np = dense_inverse_rows(A.N), nb = np / kB;
  float *R = scratch, *Cc = scratch + (size_t)kB * np;
  dense_scatter_kernel<<<(np + 255) / 256, 256, 0, st>>>(A, np, M);
  for (int k = 0; k < nb; ++k) {
    dense_pivot_kernel<<<nb, kThreads, 0, st>>>(M, np, k, R, Cc);
    dense_update_kernel<<<dim3(nb, nb), kThreads, 0, st>>>(M, np, k, R, Cc);
  }
  dense_symmetrise_kernel<<<dim3(nb, nb), kThreads, 0, st>>>(M, np);
  dense_defect_kernel<<<A.N, kThreads, 0, st>>>(A, np, M, bad);
  return cudaGetLastError();
}

}  // namespace avip
