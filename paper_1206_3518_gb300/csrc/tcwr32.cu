// W(q) . rho products of the FP32 build (step A4, the coupling block, the adjoint) on the tensor cores:
//
//   X_q[row][G] = sum_G' R_q[row][G'] W_q[G][G'],
//
// R_q the pair-density rows of one side (layout.cuh), as FP16x3 products with promoted accumulation
// (tcf16.cuh).  The rows of R and of W are split once per call into images of 8 bytes per complex value, as the FP32
// rows have.  Bound by the tensor core (24 MMAs of 56-64 cycles per 128 x 112 x 32 chunk, about 0.5 of its rate
// at 314 points) and, on small spheres, by the X rows written.  Measured against 128 x 64 register tiles on the
// FP32 pipes: fcc 8x8x8 3v4c, 128 q (314 points, 408,000 rows) 0.95 + 0.39 ms (split) against 7.09 ms; a 27 x 27
// 2v3c sheet, 128 q (115 points, 309,000 rows) 0.16 + 0.13 against 0.88 ms; fcc 4x4x4 3v3c, all 64 q 0.029 + 0.015
// against 0.081 ms: faster at every size, so there is no other route.  Error of K^d against 64 bits (2-norm): fcc
// 8x8x8 6.5e-7 (FP32 pipes 8.9e-7), fcc 6x6x6 at 12 Ha 8.3e-7 (1.1e-6), sheet 4.0e-7 (5.3e-7), fcc 4x4x4 3.6e-7
// (4.7e-7).
#include <cuda_runtime.h>

#include "internal.h"
#include "layout.cuh"
#include "tcf16.cuh"

namespace bse {
namespace {

using tcf::kTileA;
using tcf::kTKC;
using tcf::kTM;

struct WrGeo {
  int q_begin, nq, mt_max, nt_max, kc_max, n_tile, side;
  long long vbase;
};

__host__ __device__ __forceinline__ size_t a_off(const WrGeo& g, int qi, int mt) {
  return ((size_t)qi * g.mt_max + mt) * g.kc_max * (size_t)(2 * kTileA);
}
__host__ __device__ __forceinline__ size_t b_off(const WrGeo& g, int qi, int nt) {
  return ((size_t)qi * g.nt_max + nt) * g.kc_max * (size_t)(2 * g.n_tile * umma::kRow);
}

constexpr int kSplitThreads = 256;

// Rows of R_q: blockIdx.y = q of the range, GL lanes per row.
template <int GL, int NP>
__global__ __launch_bounds__(kSplitThreads) void split_rho_kernel(DevSys d, const float2* __restrict__ rho,
                                                                  unsigned char* __restrict__ img,
                                                                  float* __restrict__ inv, WrGeo g) {
  const int qi = blockIdx.y, q = g.q_begin + qi;
  const int w = side_width(d, g.side);
  const int M = (int)((d.qblk_off[q + 1] - d.qblk_off[q]) * w);
  const int row = blockIdx.x * (kSplitThreads / GL) + threadIdx.x / GL;
  const bool live = row < M;
  const float2* x = rho + (size_t)(side_rows_offset(d, q, g.side, g.vbase) + (live ? row : 0)) * d.ng_max;
  const float s = tcf::split_row<GL, NP>(x, d.ngq[q], nullptr, img + a_off(g, qi, row / kTM), 2 * kTileA, kTileA,
                                         row % kTM, live);
  if (live && threadIdx.x % GL == 0) inv[(d.qblk_off[q] - d.qblk_off[g.q_begin]) * w + row] = s;
}

// Rows of W_q.
template <int GL, int NP>
__global__ __launch_bounds__(kSplitThreads) void split_w_kernel(DevSys d, const float2* __restrict__ W,
                                                                unsigned char* __restrict__ img,
                                                                float* __restrict__ inv, WrGeo g) {
  const int qi = blockIdx.y, q = g.q_begin + qi;
  const int row = blockIdx.x * (kSplitThreads / GL) + threadIdx.x / GL;
  const bool live = row < d.ngq[q];
  const float2* x = W + ((size_t)q * d.ng_max + (live ? row : 0)) * d.ng_max;
  const uint32_t lo = (uint32_t)(g.n_tile * umma::kRow);
  const float s = tcf::split_row<GL, NP>(x, d.ngq[q], nullptr, img + b_off(g, qi, row / g.n_tile), 2 * (size_t)lo, lo,
                                         row % g.n_tile, live);
  if (live && threadIdx.x % GL == 0) inv[(size_t)qi * d.ng_max + row] = s;
}

template <int GL, int NP>
int launch_split(const DevSys& d, const void* rho, const void* W, unsigned char* As, unsigned char* Bs, float* inva,
                 float* invb, const WrGeo& g, long long max_rows, cudaStream_t st) {
  constexpr int rows = kSplitThreads / GL;
  split_rho_kernel<GL, NP><<<dim3((unsigned)((max_rows + rows - 1) / rows), g.nq), kSplitThreads, 0, st>>>(
      d, (const float2*)rho, As, inva, g);
  split_w_kernel<GL, NP><<<dim3((d.ng_max + rows - 1) / rows, g.nq), kSplitThreads, 0, st>>>(d, (const float2*)W, Bs, invb,
                                                                                          g);
  return (int)cudaGetLastError();
}

struct WrOp {
  static constexpr bool kReal = false, kConj = false, kHerm = false;
  DevSys d;
  WrGeo g;
  const unsigned char *As, *Bs;
  const float *inva, *invb;
  float2* X;
  int* status;
  long long ntiles;

  // N tiles fastest, then row tiles, then q: CTAs in flight share one q's W images and each other's R images in L2
  __device__ __forceinline__ bool tile(long long ti, tcf::Tile& o) const {
    const int nt = (int)(ti % g.nt_max);
    const long long r = ti / g.nt_max;
    const int mt = (int)(r % g.mt_max), qi = (int)(r / g.mt_max), q = g.q_begin + qi;
    const int w = side_width(d, g.side);
    const int M = (int)((d.qblk_off[q + 1] - d.qblk_off[q]) * w), NG = d.ngq[q];
    o.m0 = mt * kTM;
    o.n0 = nt * g.n_tile;
    if (o.m0 >= M || o.n0 >= NG) return false;
    o.a = As + a_off(g, qi, mt);
    o.b = Bs + b_off(g, qi, nt);
    o.a_step = 2 * kTileA;
    o.b_step = (uint32_t)(2 * g.n_tile * umma::kRow);
    o.K = NG;
    o.n = g.n_tile;
    o.mvalid = M - o.m0;
    o.nvalid = min(g.n_tile, NG - o.n0);
    o.batch = qi;
    o.row0 = (d.qblk_off[q] - d.qblk_off[g.q_begin]) * w + o.m0;
    return true;
  }

  __device__ __forceinline__ float2* row_out(const tcf::Tile& t, int row) const {
    return X + (size_t)(t.row0 + row) * d.ng_max + t.n0;
  }
  __device__ __forceinline__ float row_scale(const tcf::Tile& t, int row) const { return inva[t.row0 + row]; }
  __device__ __forceinline__ float col_scale(const tcf::Tile& t, int col) const {
    return invb[(size_t)t.batch * d.ng_max + t.n0 + col];
  }
  __device__ __forceinline__ float2 value(const tcf::Tile&, int, int, float2 s) const { return s; }
};

size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace

// Images of the R rows (w per block, at most nkpt blocks a q) and of W for a q chunk, then their inverse scales.
size_t wr32_split_bytes(const DevSys& d, long long qchunk, long long w) {
  const int n = tcf::n_tile(d.ng_max);
  const long long mt = (d.nkpt * w + kTM - 1) / kTM, nt = (d.ng_max + n - 1) / n, kc = (d.ng_max + kTKC - 1) / kTKC;
  const size_t img = (size_t)qchunk * kc * (size_t)(mt * 2 * kTileA + nt * 2 * n * umma::kRow);
  return kWsSlack + a256(img) + a256((size_t)qchunk * d.nkpt * w * sizeof(float)) +
         a256((size_t)qchunk * d.ng_max * sizeof(float));
}

int launch_gemm_wr(const DevSys& d, const void* rho, int q_begin, int q_end, long long vbase, long long max_rows,
                   const void* W, void* X, void* split_ws, int side, int* status, void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  const int w = side_width(d, side);
  WrGeo g;
  g.q_begin = q_begin;
  g.nq = q_end - q_begin;
  g.vbase = vbase;
  g.side = side;
  g.n_tile = tcf::n_tile(d.ng_max);
  g.mt_max = (int)((max_rows + kTM - 1) / kTM);
  g.nt_max = (d.ng_max + g.n_tile - 1) / g.n_tile;
  g.kc_max = (d.ng_max + kTKC - 1) / kTKC;
  if (g.nq <= 0 || g.mt_max <= 0) return 0;
  WrOp op;
  op.d = d;
  op.g = g;
  unsigned char* As = ws_base(split_ws);
  unsigned char* Bs = As + a_off(g, g.nq, 0);
  float* inva = (float*)(As + a256(a_off(g, g.nq, 0) + b_off(g, g.nq, 0)));
  float* invb = (float*)((unsigned char*)inva + a256((size_t)g.nq * d.nkpt * w * sizeof(float)));
  // lanes per row so that few idle and a row stays in registers (spheres up to 768 points; larger ones are read twice)
  const int n = d.ng_max;
  const int e = n <= 128   ? launch_split<16, 1>(d, rho, W, As, Bs, inva, invb, g, max_rows, st)
                : n <= 256 ? launch_split<16, 2>(d, rho, W, As, Bs, inva, invb, g, max_rows, st)
                : n <= 384 ? launch_split<16, 3>(d, rho, W, As, Bs, inva, invb, g, max_rows, st)
                           : launch_split<32, 3>(d, rho, W, As, Bs, inva, invb, g, max_rows, st);
  if (e) return e;
  op.As = As;
  op.Bs = Bs;
  op.inva = inva;
  op.invb = invb;
  op.X = (float2*)X;
  op.status = status;
  op.ntiles = (long long)g.nq * g.mt_max * g.nt_max;
  return tcf::launch(op, stream);
}

}  // namespace bse
