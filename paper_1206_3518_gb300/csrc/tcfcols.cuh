// Split images (tcf16.cuh) of the columns of a K-strided operand: image row g, K = k, of X[k][g].
//
// Two passes over X: the largest component of every column (colmax_kernel: atomics on the bits of the absolute value),
// then the images (split_cols_kernel: one K chunk of 32 x 64 columns per CTA, transposed in shared memory).
// Both are bound by memory: 8 bytes read per value and pass, 8 written.
//
// Src: int nbatch; int ld; bool get(int batch, const float2*& x, int& K, int& G) const (false: nothing to do).
#pragma once

#include "tcf16.cuh"

namespace bse {
namespace tcf {

constexpr int kColG = 64, kColThreads = 256, kColSlice = 512;

// mx[batch][ld] (zeroed before) = bits of max_k |component of X[k][g]|
template <class Src>
__global__ __launch_bounds__(kColThreads) void colmax_kernel(const __grid_constant__ Src src, unsigned* __restrict__ mx) {
  const float2* x;
  int K, G;
  if (!src.get(blockIdx.z, x, K, G)) return;
  const int g = blockIdx.x * kColG + (threadIdx.x & (kColG - 1)), k0 = blockIdx.y * kColSlice;
  if (blockIdx.x * kColG >= G || k0 >= K) return;
  __shared__ float red[kColThreads];
  float m = 0.f;
  if (g < G)
#pragma unroll 8
    for (int k = k0 + threadIdx.x / kColG; k < min(K, k0 + kColSlice); k += kColThreads / kColG) {
      const float2 v = x[(size_t)k * src.ld + g];
      m = fmaxf(m, fmaxf(fabsf(v.x), fabsf(v.y)));
    }
  red[threadIdx.x] = m;
  __syncthreads();
  if (threadIdx.x < kColG && g < G) {
    for (int i = 1; i < kColThreads / kColG; ++i) m = fmaxf(m, red[threadIdx.x + i * kColG]);
    if (m > 0.f) atomicMax(mx + (size_t)blockIdx.z * src.ld + g, __float_as_uint(m));
  }
}

// inverse scales from the maxima, in place
static __global__ void inv_scale_kernel(unsigned* mx, long long n) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) mx[i] = __float_as_uint(pow2(-scale_exp(__uint_as_float(mx[i]))));
}

// chunk blockIdx.y (32 k) of columns blockIdx.x * 64 ..; image of batch b at img + b batch_bytes, tiles of rows_tile
// rows, per tile kc_max chunks
template <class Src>
__global__ __launch_bounds__(kColThreads) void split_cols_kernel(const __grid_constant__ Src src,
                                                                 const float* __restrict__ inv,
                                                                 unsigned char* __restrict__ img, size_t batch_bytes,
                                                                 int rows_tile, int kc_max) {
  const float2* x;
  int K, G;
  if (!src.get(blockIdx.z, x, K, G)) return;
  const int g0 = blockIdx.x * kColG, c = blockIdx.y, k0 = c * kTKC;
  if (g0 >= G || k0 >= K) return;
  __shared__ float2 s[kTKC][kColG + 1];
  {
    const int g = g0 + (threadIdx.x & (kColG - 1));
    float2 v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int k = k0 + threadIdx.x / kColG + 4 * i;
      v[i] = g < G && k < K ? x[(size_t)k * src.ld + g] : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) s[threadIdx.x / kColG + 4 * i][threadIdx.x & (kColG - 1)] = v[i];
  }
  __syncthreads();
  const int gl = threadIdx.x >> 2, cq = threadIdx.x & 3, g = g0 + gl;
  if (g >= G) return;
  const float sc = 1.0f / inv[(size_t)blockIdx.z * src.ld + g];      // a power of two: exact
  float2 v[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float2 y = s[8 * cq + i][gl];
    v[i] = make_float2(y.x * sc, y.y * sc);
  }
  const uint32_t lo = (uint32_t)(rows_tile * umma::kRow);
  unsigned char* hi = img + (size_t)blockIdx.z * batch_bytes + ((size_t)(g / rows_tile) * kc_max + c) * (2 * (size_t)lo);
  put8(hi, hi + lo, g % rows_tile, cq, v);
}

// Bytes of the images of nbatch operands of at most K x G.
inline size_t cols_batch_bytes(int G, int K, int rows_tile) {
  return (size_t)((G + rows_tile - 1) / rows_tile) * ((K + kTKC - 1) / kTKC) * (2 * (size_t)rows_tile * umma::kRow);
}

// inv [nbatch][ld] receives the inverse scales; K, G: the largest of the batch.
template <class Src>
int split_cols(const Src& src, int K, int G, float* inv, unsigned char* img, int rows_tile, cudaStream_t st) {
  if (src.nbatch <= 0 || K <= 0 || G <= 0) return 0;
  const long long n = (long long)src.nbatch * src.ld;
  int e = (int)cudaMemsetAsync(inv, 0, (size_t)n * sizeof(float), st);
  if (e) return e;
  const int gt = (G + kColG - 1) / kColG, kc = (K + kTKC - 1) / kTKC;
  colmax_kernel<<<dim3(gt, (K + kColSlice - 1) / kColSlice, src.nbatch), kColThreads, 0, st>>>(src, (unsigned*)inv);
  inv_scale_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>((unsigned*)inv, n);
  split_cols_kernel<<<dim3(gt, kc, src.nbatch), kColThreads, 0, st>>>(src, inv, img, cols_batch_bytes(G, K, rows_tile),
                                                                     rows_tile, kc);
  return (int)cudaGetLastError();
}

}  // namespace tcf
}  // namespace bse
