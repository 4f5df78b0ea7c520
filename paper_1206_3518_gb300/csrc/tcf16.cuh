// Complex matrix products of FP32 accuracy on the 5th-generation tensor cores (FP16x3, promoted).
//
//   C[m][n] = sum_k A[m][k] B[n][k]  (or conj(A[m][k]) B[n][k]),  A and B complex64, both K-contiguous as images
//
// Splitting: every row x of an operand is scaled by a power of two that puts its largest component into
// [2^14, 2^15) and split x = hi + lo in FP16, which keeps 22 significant bits of every component down to
// 2^-17 of the row's largest (below that an absolute 2^-40 of it).  A real product is hi.hi + hi.lo + lo.hi,
// relative error ~2^-22, and the epilogue takes the scales out again (exact).
//
// Accumulation: the tensor core adds to its FP32 accumulator with truncation, measured -3.6e-8 of the sum (mean)
// after 64 products of one real sum, -3.0e-7 after 512 and -3.0e-6 after 4096, where a chain of FP32
// multiply-adds has 5e-8, 1.6e-7 and 6e-7 (rms).  So the accumulator only ever holds one K chunk (32 complex
// values, 64 real products): the correction products of the chunk are added first, while the sum is ~2^-11 of
// its final size, then the four hi.hi steps, and the epilogue warps add the chunk to FP32 registers with
// round-to-nearest while the next chunk runs in the other accumulator.  The result is as accurate as the FP32
// chain (the callers' comments have the figures).
//
// Images: per (row tile, K chunk) 128-byte rows [Re 32 | Im 32] FP16, hi rows then lo rows, 128B-swizzled K-major
// (umma.cuh).  Rows past the operand's last row are not written: they only reach accumulator rows or columns
// that are not stored.  K past the operand's length is zero.
//
// Real products (Op::kReal) use the same pipeline: 128-byte rows of 64 real K, B tiles of up to 256 rows, 12 MMAs of
// M128 N256 K16 per chunk into one accumulator of 256 columns, two stages.
//
// gemm_kernel is persistent (one CTA per SM, static round-robin over tiles): warps 0-7 promote and store (two
// warps per TMEM lane quarter, 64 columns each), warp 8 brings the images with bulk copies into a 3-stage
// ring, warp 9 issues the 24 MMAs of a chunk.  M128 x N <= 128: 64 KB per stage, two accumulators of 256 TMEM
// columns.  Every mbarrier wait is bounded (2 s); on expiry the CTA records BSE_ERR_TIMEOUT, stops issuing,
// waits (bounded) for its copies and MMAs in flight, frees its tensor memory and returns.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "internal.h"
#include "umma.cuh"

namespace bse {
namespace tcf {

constexpr int kTM = 128;                       // rows of an A tile
constexpr int kNMax = 128;                     // rows of a B tile (complex output columns), at most
constexpr int kTKC = 32;                       // complex K per chunk
constexpr int kTileA = kTM * umma::kRow;       // one split of an A tile (16 KB)
constexpr int kStages = 3;
constexpr int kStage = 2 * kTileA + 2 * kNMax * umma::kRow;
constexpr int kEpiWarps = 8, kProdWarp = 8, kMmaWarp = 9;
constexpr int kThreads = (kMmaWarp + 1) * 32;
constexpr int kAccCols = 256;                  // one accumulator: Re [0, 128), Im [128, 256)
constexpr int kRealK = 64, kRealN = 256;        // real products: K per chunk, rows of a B tile at most
constexpr int kRealStages = 2;
static_assert(kRealStages * (2 * kTileA + 2 * kRealN * umma::kRow) <= kStages * kStage, "ring");
constexpr int kXpose = 32 * 16 * 8;            // one epilogue warp's 32 x 16 complex outputs on their way out
constexpr size_t kSmem = (size_t)kStages * kStage + kEpiWarps * kXpose + 1024 + 256;

// One output tile: images of its first K chunk, bytes from chunk to chunk, K (complex, or real), B rows (a multiple of
// 16) and what the epilogue needs (origin of the tile, valid rows and columns, batch index).
struct Tile {
  const unsigned char *a, *b;
  uint32_t a_step, b_step;
  int K, n;
  int m0, n0, mvalid, nvalid, batch;
  long long row0;                              // the op's index of the tile's first row
};

// Power-of-two scale of a row whose largest |component| is m: m * 2^s in [2^14, 2^15) (below 2^-112 less).
__device__ __forceinline__ int scale_exp(float m) {
  if (!(m > 0.f)) return 0;
  const int s = 14 - ilogbf(m);                // at least -113 where m is finite
  return s > 126 ? 126 : (s < -126 ? -126 : s);
}
__device__ __forceinline__ float pow2(int s) { return __int_as_float((s + 127) << 23); }   // |s| <= 126
// x times two inverse scales, the smaller first: between a large and a small one no product leaves FP32's range that the
// result does not leave.
struct Unscale {
  float lo, hi;
  __device__ __forceinline__ Unscale(float a, float b) : lo(fminf(a, b)), hi(fmaxf(a, b)) {}
  __device__ __forceinline__ float operator()(float x) const { return x * lo * hi; }
};

// x = hi + lo in FP16 (round to nearest), two values per 32-bit word.
__device__ __forceinline__ void split_pair(float x0, float x1, uint32_t& hi, uint32_t& lo) {
  const __half2 h = __floats2half2_rn(x0, x1);
  const float2 back = __half22float2(h);
  const __half2 l = __floats2half2_rn(x0 - back.x, x1 - back.y);
  hi = *reinterpret_cast<const uint32_t*>(&h);
  lo = *reinterpret_cast<const uint32_t*>(&l);
}

// Eight consecutive K values (already scaled) into 16-byte chunks cq (Re) and 4 + cq (Im) of image row r.
__device__ __forceinline__ void put8(unsigned char* hi, unsigned char* lo, int r, int cq, const float2 (&v)[8]) {
  uint4 rh, rl, ih, il;
  split_pair(v[0].x, v[1].x, rh.x, rl.x);
  split_pair(v[2].x, v[3].x, rh.y, rl.y);
  split_pair(v[4].x, v[5].x, rh.z, rl.z);
  split_pair(v[6].x, v[7].x, rh.w, rl.w);
  split_pair(v[0].y, v[1].y, ih.x, il.x);
  split_pair(v[2].y, v[3].y, ih.y, il.y);
  split_pair(v[4].y, v[5].y, ih.z, il.z);
  split_pair(v[6].y, v[7].y, ih.w, il.w);
  *reinterpret_cast<uint4*>(hi + umma::swz(r, cq)) = rh;
  *reinterpret_cast<uint4*>(lo + umma::swz(r, cq)) = rl;
  *reinterpret_cast<uint4*>(hi + umma::swz(r, 4 + cq)) = ih;
  *reinterpret_cast<uint4*>(lo + umma::swz(r, 4 + cq)) = il;
}

// Eight values x[k0..k0+8) of a row of K (times ks[k]), zero past its end.
__device__ __forceinline__ void load8(const float2* __restrict__ x, int k0, int K, const float* __restrict__ ks,
                                      float2 (&v)[8]) {
  if (k0 + 8 <= K && (reinterpret_cast<uintptr_t>(x + k0) & 15) == 0) {
    const float4* p = reinterpret_cast<const float4*>(x + k0);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float4 u = p[i];
      v[2 * i] = make_float2(u.x, u.y);
      v[2 * i + 1] = make_float2(u.z, u.w);
    }
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = k0 + i < K ? x[k0 + i] : make_float2(0.f, 0.f);
  }
  if (ks) {
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (k0 + i < K) {
        v[i].x *= ks[k0 + i];
        v[i].y *= ks[k0 + i];
      }
  }
}

// GL lanes split one row x[0..K) (optionally times ks[k]) into image row r of its tile: chunk c at img + c step, hi
// rows of lo_off bytes then lo rows; four lanes write one 128-byte row of a chunk.  The first 8 GL NP values
// stay in registers between the search for the largest component and the split (read once; any more are read
// twice).  live: false in lanes without a row.  Returns the inverse scale 2^-s (the same in the row's lanes).
template <int GL, int NP>
__device__ __forceinline__ float split_row(const float2* __restrict__ x, int K, const float* __restrict__ ks,
                                           unsigned char* img, size_t step, uint32_t lo_off, int r, bool live) {
  const int lane = threadIdx.x & (GL - 1), nt = live ? 4 * ((K + kTKC - 1) / kTKC) : 0, Kr = live ? K : 0;
  float2 v[NP][8];
  float m = 0.f;
  auto largest = [&](const float2 (&u)[8]) {
#pragma unroll
    for (int i = 0; i < 8; ++i) m = fmaxf(m, fmaxf(fabsf(u[i].x), fabsf(u[i].y)));
  };
#pragma unroll
  for (int p = 0; p < NP; ++p) {
    load8(x, 8 * (lane + GL * p), Kr, ks, v[p]);
    largest(v[p]);
  }
  for (int t = lane + GL * NP; t < nt; t += GL) {
    float2 u[8];
    load8(x, 8 * t, Kr, ks, u);
    largest(u);
  }
#pragma unroll
  for (int o = GL / 2; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  const int e = scale_exp(m);
  const float sc = pow2(e);
  auto put = [&](int t, float2 (&u)[8]) {
#pragma unroll
    for (int i = 0; i < 8; ++i) u[i] = make_float2(u[i].x * sc, u[i].y * sc);
    unsigned char* hi = img + (size_t)(t >> 2) * step;
    put8(hi, hi + lo_off, r, t & 3, u);
  };
#pragma unroll
  for (int p = 0; p < NP; ++p)
    if (lane + GL * p < nt) put(lane + GL * p, v[p]);
  for (int t = lane + GL * NP; t < nt; t += GL) {
    float2 u[8];
    load8(x, 8 * t, Kr, ks, u);
    put(t, u);
  }
  return pow2(-e);
}

// Instruction descriptor: D f32, A/B f16, both K-major, M = 128, N = n (bit 13 negates A).
__host__ __device__ constexpr uint32_t idesc_f16(int n) {
  return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kTM >> 4) << 24);
}

// The 12 NKK MMAs of one chunk (descriptors of the hi tiles, offsets of the lo tiles in 16-byte units): corrections
// first, then hi.hi; Re before Im within each (a change of accumulator costs 5 cycles).  CONJ: conj(A) B.
template <bool CONJ, int NKK>
__device__ __forceinline__ void chunk_mmas(uint32_t d_re, uint32_t d_im, uint64_t da, uint32_t a_lo, uint64_t db,
                                           uint32_t b_lo, uint32_t idesc) {
  const uint32_t neg = idesc | umma::kNegA;
#pragma unroll
  for (int im = 0; im < 2; ++im) {
    const uint32_t d = im ? d_im : d_re, sign = (im != 0) == CONJ ? neg : idesc;   // of the product with Im A
    const uint32_t b0 = im ? 4u : 0u, b1 = 4u - b0;                            // plane of B met by Re A, by Im A
#pragma unroll
    for (int s = 0; s < 3; ++s)                  // hi.lo and lo.hi, then hi.hi
#pragma unroll
      for (int kk = NKK - 1; kk >= 0; --kk) {
        const uint64_t pa = da + (s == (CONJ ? 0 : 1) ? a_lo : 0u) + (uint32_t)kk * 2u;
        const uint64_t pb = db + (s == (CONJ ? 1 : 0) ? b_lo : 0u) + (uint32_t)kk * 2u;
        umma::mma_f16(d, pa, pb + b0, idesc, (s != 0 || kk != NKK - 1) ? 1u : 0u);
        umma::mma_f16(d, pa + 4u, pb + b1, sign, 1u);
      }
  }
}

// The 3 nkk MMAs of one chunk of a real product.
__device__ __forceinline__ void chunk_mmas_real(uint32_t d, uint64_t da, uint32_t a_lo, uint64_t db, uint32_t b_lo, int nkk,
                                                uint32_t idesc) {
#pragma unroll
  for (int s = 0; s < 3; ++s)                    // hi.lo, lo.hi, hi.hi
#pragma unroll
    for (int kk = 0; kk < 4; ++kk)
      if (kk < nkk)
        umma::mma_f16(d, da + (s == 1 ? a_lo : 0u) + (uint32_t)kk * 2u, db + (s == 0 ? b_lo : 0u) + (uint32_t)kk * 2u,
                       idesc, (s | kk) != 0 ? 1u : 0u);
}

// The MMAs of a complex chunk of NKK K16 groups with the A planes in tensor memory at columns a + 0 (Re hi), a + 8 (Im
// hi), a + 16 (Re lo), a + 24 (Im lo) of the first group, + 32 per further one (two FP16 per 32-bit column, lane =
// row), B panels of two groups b_sub apart; A as it is (no conjugation).
template <int NKK>
__device__ __forceinline__ void chunk_mmas_ts(uint32_t d_re, uint32_t d_im, uint32_t a, uint64_t db, uint32_t b_lo,
                                              uint32_t b_sub, uint32_t idesc) {
  const uint32_t neg = idesc | umma::kNegA;
#pragma unroll
  for (int im = 0; im < 2; ++im) {
    const uint32_t d = im ? d_im : d_re, sign = im ? idesc : neg;
    const uint32_t b0 = im ? 4u : 0u, b1 = 4u - b0;
#pragma unroll
    for (int s = 0; s < 3; ++s)                  // hi.lo, lo.hi, hi.hi
#pragma unroll
      for (int kk = NKK - 1; kk >= 0; --kk) {
        const uint32_t pa = a + (uint32_t)kk * 32u + (s == 1 ? 16u : 0u);
        const uint64_t pb = db + (s == 0 ? b_lo : 0u) + (uint32_t)(kk >> 1) * b_sub + (uint32_t)(kk & 1) * 2u;
        umma::mma_f16_ts(d, pa, pb + b0, idesc, (s != 0 || kk != NKK - 1) ? 1u : 0u);
        umma::mma_f16_ts(d, pa + 8u, pb + b1, sign, 1u);
      }
  }
}

__device__ __forceinline__ void fail_now(volatile int* fail, int* status) {
  *fail = 1;
  atomicCAS(status, 0, (int)BSE_ERR_TIMEOUT);
}

// Op: long long ntiles; int* status; static constexpr bool kReal, kConj, kHerm (tiles m0 <= n0 of a Hermitian
// result: the upper triangle is stored with its mirror image, float2* mirror_out(...)); bool tile(long long t, Tile&)
// (false: nothing to do); float2* row_out(const Tile&, int row) the address of column 0 of a row of the tile; float
// row_scale(const Tile&, int row), col_scale(const Tile&, int col) the inverse scales; float2 value(const Tile&, int
// row, int col, float2 sum) the output from the unscaled sum (real: float* row_out, no value()).  Outputs go out
// through shared memory, 16 columns at a time, so that eight lanes write 128 contiguous bytes of a row (rows stored lane by lane cost 2.8 times the
// time of the whole product at 115 columns: 294 us against 106 us without stores).
template <class Op>
__global__ __launch_bounds__(kThreads, 1) void gemm_kernel(const __grid_constant__ Op op) {
  constexpr bool R = Op::kReal;
  constexpr int kChunk = R ? kRealK : kTKC, kRing = R ? kRealStages : kStages;
  constexpr int kStageB = 2 * kTileA + 2 * (R ? kRealN : kNMax) * umma::kRow;
  extern __shared__ __align__(1024) unsigned char tcf_smem_raw[];
  unsigned char* sm = (unsigned char*)(((uintptr_t)tcf_smem_raw + 1023) & ~(uintptr_t)1023);
  unsigned char* xpose = sm + kStages * kStage;   // after the ring (the larger of the two)
  uint64_t* full = (uint64_t*)(xpose + kEpiWarps * kXpose);   // [3] stage landed
  uint64_t* empty = full + kStages;                       // [3] MMAs done with the stage
  uint64_t* tfull = empty + kStages;                      // [2] accumulator holds a chunk
  uint64_t* tempty = tfull + 2;                           // [2] accumulator promoted
  uint64_t* drain = tempty + 2;                           // all MMAs of this CTA complete
  uint32_t* tmem_slot = (uint32_t*)(drain + 1);
  volatile int* fail = (volatile int*)(tmem_slot + 1);
  volatile unsigned* issued = (volatile unsigned*)(tmem_slot + 2);
  volatile unsigned* consumed = (volatile unsigned*)(tmem_slot + 3);
  const int tid = threadIdx.x, warp = umma::uniform(tid >> 5), lane = tid & 31;
  using umma::smem_u32;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(2 * kAccCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 32) {
    for (int i = 0; i < kRing; ++i) {
      umma::mbar_init(smem_u32(full + i), 1);
      umma::mbar_init(smem_u32(empty + i), 1);
    }
    for (int i = 0; i < 2; ++i) {
      umma::mbar_init(smem_u32(tfull + i), 1);
      umma::mbar_init(smem_u32(tempty + i), kEpiWarps);
    }
    umma::mbar_init(smem_u32(drain), 1);
    *fail = 0;
    *issued = 0;
    *consumed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  if (warp == kProdWarp) {
    if (lane == 0) {
      unsigned c = 0;
      Tile t;
      for (long long ti = blockIdx.x; ti < op.ntiles && !*fail; ti += gridDim.x) {
        if (!op.tile(ti, t)) continue;
        const int nch = (t.K + kChunk - 1) / kChunk;
        const uint32_t bbytes = (uint32_t)(2 * t.n * umma::kRow);
        for (int kc = 0; kc < nch; ++kc, ++c) {
          const int st = (int)(c % kRing);
          if (c >= kRing && !umma::mbar_wait(smem_u32(empty + st), ((c / kRing) - 1) & 1u)) {
            fail_now(fail, op.status);
            break;
          }
          if (*fail) break;
          const uint32_t base = smem_u32(sm + st * kStageB);
          umma::mbar_arrive_expect_tx(smem_u32(full + st), (uint32_t)(2 * kTileA) + bbytes);
          umma::bulk_g2s(base, t.a + (size_t)kc * t.a_step, 2 * kTileA, smem_u32(full + st));
          umma::bulk_g2s(base + 2 * kTileA, t.b + (size_t)kc * t.b_step, bbytes, smem_u32(full + st));
          *issued = c + 1;
        }
      }
    }
  } else if (warp == kMmaWarp) {                   // the whole warp runs the loop, one lane issues
    const bool leader = umma::elect_one();
    const uint64_t d0 = umma::smem_desc(umma::uniform(smem_u32(sm)));
    unsigned c = 0;
    Tile t;
    bool ok = true;
    for (long long ti = blockIdx.x; ti < op.ntiles && ok; ti += gridDim.x) {
      if (!op.tile(ti, t)) continue;
      const int K = umma::uniform(t.K), n = umma::uniform(t.n), nch = (K + kChunk - 1) / kChunk;
      const uint32_t idesc = idesc_f16(n), b_lo = (uint32_t)(n * umma::kRow) >> 4;
      for (int kc = 0; kc < nch; ++kc, ++c) {
        const int st = (int)(c % kRing), buf = (int)(c & 1u);
        ok = umma::uniform((c < 2 || umma::mbar_wait(smem_u32(tempty + buf), ((c >> 1) - 1) & 1u)) &&
                           umma::mbar_wait(smem_u32(full + st), (c / kRing) & 1u) && !*fail);
        if (!ok) {
          if (leader) fail_now(fail, op.status);
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint64_t da = d0 + (uint64_t)((st * kStageB) >> 4), db = da + (uint64_t)((2 * kTileA) >> 4);
        const uint32_t d_re = umma::uniform(tmem + (uint32_t)(buf * kAccCols));
        if (leader) {
          if (R)
            chunk_mmas_real(d_re, da, (uint32_t)(kTileA >> 4), db, b_lo, (K - kc * kChunk + 15) / 16, idesc);
          else if (K - kc * kTKC > 16)
            chunk_mmas<Op::kConj, 2>(d_re, d_re + 128u, da, (uint32_t)(kTileA >> 4), db, b_lo, idesc);
          else
            chunk_mmas<Op::kConj, 1>(d_re, d_re + 128u, da, (uint32_t)(kTileA >> 4), db, b_lo, idesc);
          umma::mma_commit(smem_u32(empty + st));
          umma::mma_commit(smem_u32(tfull + buf));
          *consumed = c + 1;
        }
        __syncwarp();
      }
    }
    if (leader) {
      umma::mma_commit(smem_u32(drain));           // tracks every MMA issued above
      if (!umma::mbar_wait(smem_u32(drain), 0u)) fail_now(fail, op.status);
    }
    __syncwarp();
  } else {                                         // promote: lanes 32 (warp & 3) .., columns 64 (warp >> 2) ..
    const int c0 = (warp >> 2) * 64;
    const uint32_t lane_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c0;
    unsigned c = 0;
    Tile t;
    bool ok = true;
    for (long long ti = blockIdx.x; ti < op.ntiles && ok; ti += gridDim.x) {
      if (!op.tile(ti, t)) continue;
      const int nch = (t.K + kChunk - 1) / kChunk;
      float re[4][16], im[4][16];
#pragma unroll
      for (int g = 0; g < 4; ++g)
#pragma unroll
        for (int i = 0; i < 16; ++i) re[g][i] = im[g][i] = 0.f;
      for (int kc = 0; kc < nch; ++kc, ++c) {
        const int buf = (int)(c & 1u);
        int good = 1;
        if (lane == 0) {
          good = umma::mbar_wait(smem_u32(tfull + buf), (c >> 1) & 1u) ? 1 : 0;
          if (!good) fail_now(fail, op.status);
        }
        good = __shfl_sync(0xffffffffu, good, 0);
        __syncwarp();                              // orders lane 0's acquire before the warp's loads (a shuffle does not)
        if (!good) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t base = lane_addr + (uint32_t)(buf * kAccCols);
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          if (!R && c0 + 16 * g >= t.n) break;
          uint32_t v[16];
          umma::tmem_ld16(base + 16u * g, v);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int i = 0; i < 16; ++i) re[g][i] += __uint_as_float(v[i]);
          umma::tmem_ld16(base + 128u + 16u * g, v);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int i = 0; i < 16; ++i) im[g][i] += __uint_as_float(v[i]);
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) umma::mbar_arrive(smem_u32(tempty + buf));
      }
      if (ok) {
        unsigned char* xp = xpose + warp * kXpose;
        const int row = (warp & 3) * 32 + lane;
        const float sa = row < t.mvalid ? op.row_scale(t, row) : 0.f;
        if constexpr (R) {                         // columns c0 + 16 g.. (re) and 128 + c0 + 16 g.. (im), 16 at a time
#pragma unroll
          for (int g = 0; g < 8; ++g) {
            const int cb = (g < 4 ? 0 : 128) + c0 + 16 * (g & 3);
            if (cb >= t.nvalid) continue;
            const float(&v)[16] = g < 4 ? re[g & 3] : im[g & 3];
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 4; ++i)
              *reinterpret_cast<float4*>(xp + lane * 64 + ((i ^ ((lane >> 1) & 3)) << 4)) =
                  make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
            __syncwarp();
            const int j = lane & 3, col = cb + 4 * j;
            float s[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) s[i] = col + i < t.nvalid ? op.col_scale(t, col + i) : 0.f;
#pragma unroll 2
            for (int r8 = 0; r8 < 4; ++r8) {
              const int rl = r8 * 8 + (lane >> 2), ro = (warp & 3) * 32 + rl;
              const float sr = __shfl_sync(0xffffffffu, sa, rl);
              if (ro >= t.mvalid || col >= t.nvalid) continue;
              const float4 u = *reinterpret_cast<const float4*>(xp + rl * 64 + ((j ^ ((rl >> 1) & 3)) << 4));
              float* out = op.row_out(t, ro) + col;
              const float w[4] = {Unscale(sr, s[0])(u.x), Unscale(sr, s[1])(u.y), Unscale(sr, s[2])(u.z), Unscale(sr, s[3])(u.w)};
              if (col + 3 < t.nvalid && (reinterpret_cast<uintptr_t>(out) & 15) == 0) {
                *reinterpret_cast<float4*>(out) = make_float4(w[0], w[1], w[2], w[3]);
              } else {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                  if (col + i < t.nvalid) out[i] = w[i];
              }
            }
          }
        } else {
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          if (c0 + 16 * g >= t.nvalid) break;
          __syncwarp();
#pragma unroll
          for (int i = 0; i < 8; ++i)
            *reinterpret_cast<float4*>(xp + lane * 128 + ((i ^ (lane & 7)) << 4)) =
                make_float4(re[g][2 * i], im[g][2 * i], re[g][2 * i + 1], im[g][2 * i + 1]);
          __syncwarp();
          const int j = lane & 7, col = c0 + 16 * g + 2 * j;
          const float s0 = col < t.nvalid ? op.col_scale(t, col) : 0.f;
          const float s1 = col + 1 < t.nvalid ? op.col_scale(t, col + 1) : 0.f;
#pragma unroll 2
          for (int r4 = 0; r4 < 8; ++r4) {
            const int rl = r4 * 4 + (lane >> 3), ro = (warp & 3) * 32 + rl;
            const float sr = __shfl_sync(0xffffffffu, sa, rl);
            if (ro >= t.mvalid || col >= t.nvalid) continue;
            float4 v = *reinterpret_cast<const float4*>(xp + rl * 128 + ((j ^ (rl & 7)) << 4));
            const Unscale u0(sr, s0), u1(sr, s1);
            v = make_float4(u0(v.x), u0(v.y), u1(v.z), u1(v.w));
            float2* out = op.row_out(t, ro) + col;
            if constexpr (Op::kHerm) {             // upper triangle, and its mirror image
#pragma unroll
              for (int i = 0; i < 2; ++i) {
                if (col + i >= t.nvalid || t.m0 + ro > t.n0 + col + i) continue;
                float2 y = op.value(t, ro, col + i, i ? make_float2(v.z, v.w) : make_float2(v.x, v.y));
                if (t.m0 + ro == t.n0 + col + i) y.y = 0.f;
                out[i] = y;
                if (t.m0 + ro != t.n0 + col + i) *op.mirror_out(t, ro, col + i) = make_float2(y.x, -y.y);
              }
              continue;
            }
            const float2 y0 = op.value(t, ro, col, make_float2(v.x, v.y));
            if (col + 1 < t.nvalid) {
              const float2 y1 = op.value(t, ro, col + 1, make_float2(v.z, v.w));
              if ((reinterpret_cast<uintptr_t>(out) & 15) == 0) {
                *reinterpret_cast<float4*>(out) = make_float4(y0.x, y0.y, y1.x, y1.y);
              } else {
                out[0] = y0;
                out[1] = y1;
              }
            } else {
              out[0] = y0;
            }
          }
        }
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (tid == 0) {                                  // copies still in flight after a failure
    for (unsigned c = *consumed; c < *issued; ++c)
      if (!umma::mbar_wait(smem_u32(full + c % kRing), (c / kRing) & 1u)) break;
  }
  __syncthreads();
  if (warp == 0) {
    __syncwarp();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * kAccCols) : "memory");
  }
}

// Rows of a B tile for n columns: ceil(n / ceil(n / 128)) rounded up to 16.
inline int n_tile(int n) {
  const int nt = (n + kNMax - 1) / kNMax;
  return ((n + nt - 1) / nt + 15) / 16 * 16;
}

template <class Op>
int launch(const Op& op, void* stream) {
  if (op.ntiles <= 0) return 0;
  int dev = 0, sms = 0;
  int e = (int)cudaGetDevice(&dev);
  if (e) return e;
  if ((e = (int)cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev))) return e;
  if ((e = (int)cudaFuncSetAttribute((const void*)gemm_kernel<Op>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)kSmem)))
    return e;
  const int grid = (int)(op.ntiles < sms ? op.ntiles : sms);
  gemm_kernel<Op><<<grid, kThreads, kSmem, (cudaStream_t)stream>>>(op);
  return (int)cudaGetLastError();
}

}  // namespace tcf
}  // namespace bse
