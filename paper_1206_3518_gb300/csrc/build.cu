// Kernel contractions and Hamiltonian assembly, CUDA-core FP32 form (steps A3-A5).
//
// Eq. kernel (TDA, singlet):  H = diag(e_c + Delta - e_v) + 2 K^x - K^d
//   K^x_SS' = (1/(Omega Nk)) sum_{G != 0} conj(rho_vc^{kk}(G)) vbar(G) rho_v'c'^{k'k'}(G)   (Eq. V_eh)
//   K^d_SS' = (1/(Omega Nk)) sum_{G,G'} conj(rho_vv'^{kk'}(G)) W_GG'(q) rho_cc'^{kk'}(G')  (Eq. W_SS)
//
// init_kernel   : 2K^x + diag on every tile that touches the upper block triangle; the
//                 exchange scale sqrt(2 vbar/(Omega Nk)) is applied to both operands (a build
//                 without a workspace at this step; with one, tcgram32.cu).
// W.rho         : per q, X = W(q) R for the smaller band side (grouped over the q chunk), stored as
//                 X^T rows [col][G] (G contiguous); on the tensor cores (tcwr32.cu, FP32 accuracy).
// block_kernel  : per upper block (k <= k'), M = X^H R of the other side (K = NG_q),
//                 H_kk' = H_kk' - M/(Omega Nk) and the mirror H_k'k = H_kk'^H;
//                 diagonal blocks become (B + B^H)/2.
// init_kernel uses the tiled FP32 complex "NT" core of gemm_tile.cuh: C[m][n] =
// sum_k opA(A[m][k]) B[n][k] with both operands K-contiguous.
#include <cuda_runtime.h>

#include "gemm_tile.cuh"
#include "internal.h"
#include "layout.cuh"

namespace bse {
namespace {

using gemm::BM;
using gemm::BN;
constexpr int kGemmThreads = gemm::kThreads;

__device__ __forceinline__ int kpt_of_pair(const DevSys& d, int S) { return S / (d.nv * d.nc); }

// H[S][S'] = 2 K^x + delta_SS' (e_c + Delta - e_v) on tiles touching k(S) <= k(S').
__global__ __launch_bounds__(kGemmThreads) void init_kernel(DevSys d, const float2* __restrict__ rho_x,
                                                            const double* __restrict__ e, double delta,
                                                            float2* __restrict__ H) {
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  if (m0 >= d.dim || n0 >= d.dim) return;
  if (kpt_of_pair(d, m0) > kpt_of_pair(d, min(n0 + BN, d.dim) - 1)) return;   // strictly lower block triangle
  __shared__ gemm::Smem sm;
  float2 acc[4][4];
  gemm::tile<true, true, true, false, true>(rho_x, d.ng_max, d.dim, rho_x, d.ng_max, d.dim, d.ng0, m0, n0, sm, acc,
                                            d.xscale);
  const int tm = threadIdx.x / 16, tn = threadIdx.x % 16;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int S = m0 + tm * 4 + i;
    if (S >= d.dim) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int S2 = n0 + tn * 4 + j;
      if (S2 >= d.dim) continue;
      float2 v = acc[i][j];
      if (S == S2) {
        const int ic = S % d.nc, iv = (S / d.nc) % d.nv, k = S / (d.nv * d.nc);
        v.x += (float)(e[(size_t)k * d.nb + d.nv + ic] + delta - e[(size_t)k * d.nb + iv]);
      }
      H[(size_t)S * d.dim + S2] = v;
    }
  }
}

constexpr int kBlkThreads = 256, KC = 32;

constexpr int kBlkWarps = 4;             // block_kernel: blocks (warps) per CTA
constexpr int kBlkStages = 3;            // K steps in a warp's ring: one in use, two in flight
constexpr int kBlkK = 16;                // complex K values per step: 128 bytes of a row
constexpr int kBlkRow = kBlkK + 2;       // entries of a ring row: 16-byte rows four banks apart

__host__ __device__ constexpr int blk_warp_bytes(int rows) { return kBlkStages * rows * kBlkRow * (int)sizeof(float2); }

// `bytes` of 16 (past L1) or of 8 from global to shared memory, the rest zero.
__device__ __forceinline__ void cp_async16(float2* dst, const float2* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void cp_async8(float2* dst, const float2* src, int bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(bytes)
               : "memory");
}

// Per upper block: M[a][c] = sum_G conj(L[a][G]) Rr[c][G], a = (v,v'), c = (c,c');
// side V: L = X (= W R_v), Rr = R_c;  side C: L = R_v, Rr = X (= W R_c).
// One warp per block, so that no barrier couples blocks of different q, and a ring of three K steps per warp filled
// with 16-byte asynchronous copies past L1 (8-byte ones, which go through L1, hold a line of it each while in flight).
// LI x (32 / LI) lanes with a PI x PJ patch each, a = i + LI x, c = j + LJ y; the patch is the smallest that covers
// nv^2 x nc^2 (lanes beyond it read the last row and store nothing).  Each entry is the same chain of fused
// multiply-adds over G whatever the patch.  EVEN: every row starts on a 16-byte boundary (two values per load).
// Bound by HBM (every density and X row is read once) and, close to it, by shared-memory reads (LDS of PI + PJ values for
// 4 PI PJ multiply-adds).  Measured, all q (ms; before: four blocks per CTA of 256 threads, 2 x 2 patches, loads through
// registers with two CTA barriers a step): fcc 8x8x8 3v4c 1.71 (2.90; 8.2 GB, 0.72 of the copy rate), fcc 12x12x12 4v4c
// 51.8 (56), 27 x 27 sheet 2v3c 0.91 (2.3).
template <int LI, int PI, int PJ, bool EVEN>
__global__ __launch_bounds__(kBlkWarps * 32) void block_kernel(DevSys d, const float2* __restrict__ rho_dir,
                                                              const float2* __restrict__ X, float2* __restrict__ H,
                                                              int q_begin, long long vbase, int side_c,
                                                              long long b_count) {
  extern __shared__ __align__(16) unsigned char blk_smem[];
  constexpr int LJ = 32 / LI;
  const int lane = threadIdx.x % 32;
  const long long bi = (long long)blockIdx.x * kBlkWarps + threadIdx.x / 32;
  if (bi >= b_count) return;                          // whole warps; the kernel has no CTA barrier
  const int nv2 = d.nv * d.nv, nc2 = d.nc * d.nc, rows = nv2 + nc2;
  float2* ring = reinterpret_cast<float2*>(blk_smem + (threadIdx.x / 32) * blk_warp_bytes(rows));
  const long long b0 = d.qblk_off[q_begin];
  const long long b = b0 + bi;
  const int4 blk = d.blocks[b];
  const int k = blk.x, k2 = blk.y, q = blk.z;
  const long long qb = d.qblk_off[q];
  const long long nblk = d.qblk_off[q + 1] - qb;
  const long long local = b - qb;
  const long long vbase_q = d.qvec_off[q] - vbase;
  const float2* Rv = rho_dir + (size_t)(vbase_q + local * nv2) * d.ng_max;
  const float2* Rc = rho_dir + (size_t)(vbase_q + nblk * nv2 + local * nc2) * d.ng_max;
  const int w = side_c ? nc2 : nv2;
  const float2* Xb = X + (size_t)((qb - b0 + local) * w) * d.ng_max;
  const float2* L = side_c ? Rv : Xb;
  const float2* R = side_c ? Xb : Rc;
  const int NG = d.ngq[q], steps = (NG + kBlkK - 1) / kBlkK;

  // Eight lanes per row, four rows at once.  Entry e of a step lies in slot e + odd(row), so that the 16-byte copies keep
  // their alignment in rows that start on an odd multiple of eight bytes; there the eighth lane brings the first and
  // the last entry.  A lane's rows are a multiple of four rows apart and share that parity.
  const int l8 = lane & 7, r0 = lane >> 3;
  auto load_rows = [&](const float2* src, float2* dst, int n, int left) {
    src += (size_t)r0 * d.ng_max;
    const int odd = EVEN ? 0 : (int)(reinterpret_cast<uintptr_t>(src) >> 3) & 1;
    const int e = odd + 2 * l8;
    dst += r0 * kBlkRow;
    for (int r = r0; r < n; r += 4) {
      if (!EVEN && odd && l8 == 7) {
        const bool last = left > kBlkK - 1;
        cp_async8(dst + 1, src, 8);
        cp_async8(dst + kBlkK, last ? src + kBlkK - 1 : src, last ? 8 : 0);
      } else {
        const int m = min(max(left - e, 0), 2);
        cp_async16(dst + odd + e, src + (m > 0 ? e : -odd), 8 * m);
      }
      src += 4 * (size_t)d.ng_max;
      dst += 4 * kBlkRow;
    }
  };
  auto load = [&](int it) {
    if (it < steps) {
      float2* dst = ring + (it % kBlkStages) * rows * kBlkRow;
      load_rows(L + it * kBlkK, dst, nv2, NG - it * kBlkK);
      load_rows(R + it * kBlkK, dst + nv2 * kBlkRow, nc2, NG - it * kBlkK);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };

  const int i0 = lane / LJ, j0 = lane % LJ;
  int lo[PI], ro[PJ];
  auto slot = [&](const float2* row, int r) {
    return r * kBlkRow + (EVEN ? 0 : (int)(reinterpret_cast<uintptr_t>(row) >> 3) & 1);
  };
#pragma unroll
  for (int x = 0; x < PI; ++x) {
    const int r = min(i0 + LI * x, nv2 - 1);
    lo[x] = slot(L + (size_t)r * d.ng_max, r);
  }
#pragma unroll
  for (int y = 0; y < PJ; ++y) {
    const int r = min(j0 + LJ * y, nc2 - 1);
    ro[y] = slot(R + (size_t)r * d.ng_max, nv2 + r);
  }
  float2 acc[PI][PJ];
#pragma unroll
  for (int x = 0; x < PI; ++x)
#pragma unroll
    for (int y = 0; y < PJ; ++y) acc[x][y] = make_float2(0.f, 0.f);

#pragma unroll
  for (int s = 0; s < kBlkStages - 1; ++s) load(s);
  for (int it = 0; it < steps; ++it) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kBlkStages - 2) : "memory");
    __syncwarp();                                     // step it has landed; all lanes are done with step it - 1
    load(it + kBlkStages - 1);
    const float2* st = ring + (it % kBlkStages) * rows * kBlkRow;
    auto mac = [&](const float2 (&l)[PI], const float2 (&r)[PJ]) {
#pragma unroll
      for (int x = 0; x < PI; ++x)
#pragma unroll
        for (int y = 0; y < PJ; ++y) {
          acc[x][y].x = fmaf(l[x].x, r[y].x, fmaf(l[x].y, r[y].y, acc[x][y].x));         // conj(l) r
          acc[x][y].y = fmaf(l[x].x, r[y].y, fmaf(-l[x].y, r[y].x, acc[x][y].y));
        }
    };
    if constexpr (EVEN) {
#pragma unroll 4
      for (int g = 0; g < kBlkK; g += 2) {
        float2 l0[PI], l1[PI], r0_[PJ], r1[PJ];
#pragma unroll
        for (int x = 0; x < PI; ++x) {
          const float4 v = *reinterpret_cast<const float4*>(st + lo[x] + g);
          l0[x] = make_float2(v.x, v.y);
          l1[x] = make_float2(v.z, v.w);
        }
#pragma unroll
        for (int y = 0; y < PJ; ++y) {
          const float4 v = *reinterpret_cast<const float4*>(st + ro[y] + g);
          r0_[y] = make_float2(v.x, v.y);
          r1[y] = make_float2(v.z, v.w);
        }
        mac(l0, r0_);
        mac(l1, r1);
      }
    } else {
#pragma unroll 8
      for (int g = 0; g < kBlkK; ++g) {
        float2 l[PI], r[PJ];
#pragma unroll
        for (int x = 0; x < PI; ++x) l[x] = st[lo[x] + g];
#pragma unroll
        for (int y = 0; y < PJ; ++y) r[y] = st[ro[y] + g];
        mac(l, r);
      }
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncwarp();

  const int nv = d.nv, nc = d.nc, nvc = nv * nc;
  const float nrm = (float)d.norm;
  float2* Bs = ring;                                  // the diagonal block: nvc (nvc + 1) <= 54 (nv^2 + nc^2)
#pragma unroll
  for (int x = 0; x < PI; ++x)
#pragma unroll
    for (int y = 0; y < PJ; ++y) {
      const int a = i0 + LI * x, c = j0 + LJ * y;
      if (a >= nv2 || c >= nc2) continue;
      const int row = (a / nv) * nc + c / nc;          // (k, v, c) local
      const int col = (a % nv) * nc + c % nc;          // (k', v', c') local
      const size_t hij = (size_t)(k * nvc + row) * d.dim + (size_t)k2 * nvc + col;
      const float2 h = H[hij];
      const float2 val = make_float2(h.x - nrm * acc[x][y].x, h.y - nrm * acc[x][y].y);
      acc[x][y] = val;
      if (k != k2) {
        H[hij] = val;
        H[(size_t)(k2 * nvc + col) * d.dim + (size_t)k * nvc + row] = make_float2(val.x, -val.y);
      } else {
        Bs[row * (nvc + 1) + col] = val;
      }
    }
  if (k == k2) {
    __syncwarp();
#pragma unroll
    for (int x = 0; x < PI; ++x)
#pragma unroll
      for (int y = 0; y < PJ; ++y) {
        const int a = i0 + LI * x, c = j0 + LJ * y;
        if (a >= nv2 || c >= nc2) continue;
        const int row = (a / nv) * nc + c / nc, col = (a % nv) * nc + c % nc;
        const float2 o = Bs[col * (nvc + 1) + row];
        H[(size_t)(k * nvc + row) * d.dim + (size_t)k * nvc + col] =
            make_float2(0.5f * (acc[x][y].x + o.x), 0.5f * (acc[x][y].y - o.y));
      }
  }
}

template <int LI, int PI, int PJ>
int launch_block(const DevSys& d, const float2* rho, const float2* X, float2* H, int q_begin, long long vbase,
                 int side_c, long long b_count, cudaStream_t st) {
  const int smem = kBlkWarps * blk_warp_bytes(d.nv * d.nv + d.nc * d.nc);       // at most 54 KB
  const bool even = d.ng_max % 2 == 0 && ((reinterpret_cast<uintptr_t>(rho) | reinterpret_cast<uintptr_t>(X)) & 15) == 0;
  auto kernel = even ? block_kernel<LI, PI, PJ, true> : block_kernel<LI, PI, PJ, false>;
  if (int e = allow_smem((const void*)kernel)) return e;
  kernel<<<(unsigned)((b_count + kBlkWarps - 1) / kBlkWarps), kBlkWarps * 32, smem, st>>>(d, rho, X, H, q_begin, vbase,
                                                                                         side_c, b_count);
  return (int)cudaGetLastError();
}

// The longer side takes the eight lanes; nv^2 and nc^2 are 1, 4, 9 or 16.
int launch_blocks(const DevSys& d, const float2* rho, const float2* X, float2* H, int q_begin, long long vbase,
                  int side_c, long long b_count, cudaStream_t st) {
  const int nv = d.nv, nc = d.nc;
  if (nv <= nc) {
    if (nc <= 2) return launch_block<4, 1, 1>(d, rho, X, H, q_begin, vbase, side_c, b_count, st);
    if (nv <= 2) return launch_block<4, 1, 2>(d, rho, X, H, q_begin, vbase, side_c, b_count, st);
    if (nv == 3) return launch_block<4, 3, 2>(d, rho, X, H, q_begin, vbase, side_c, b_count, st);
    return launch_block<4, 4, 2>(d, rho, X, H, q_begin, vbase, side_c, b_count, st);
  }
  if (nv <= 2) return launch_block<8, 1, 1>(d, rho, X, H, q_begin, vbase, side_c, b_count, st);
  if (nc <= 2) return launch_block<8, 2, 1>(d, rho, X, H, q_begin, vbase, side_c, b_count, st);
  return launch_block<8, 2, 3>(d, rho, X, H, q_begin, vbase, side_c, b_count, st);
}

// Lower blocks from the upper ones, H_k'k = H_kk'^H, and diagonal blocks (B + B^H)/2 (for a build
// without the direct term, which otherwise does this in its epilogue).
__global__ void mirror_kernel(DevSys d, float2* __restrict__ H) {
  const long long n = (long long)d.dim * d.dim;
  const int nvc = d.nv * d.nc;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const int S = (int)(i / d.dim), S2 = (int)(i - (long long)S * d.dim);
    const int k = S / nvc, k2 = S2 / nvc;
    if (k > k2) {
      const float2 u = H[(size_t)S2 * d.dim + S];
      H[i] = make_float2(u.x, -u.y);
    } else if (k == k2 && S < S2) {
      const float2 a = H[i], b = H[(size_t)S2 * d.dim + S];
      const float2 m = make_float2(0.5f * (a.x + b.x), 0.5f * (a.y - b.y));
      H[i] = m;
      H[(size_t)S2 * d.dim + S] = make_float2(m.x, -m.y);
    } else if (S == S2) {
      H[i].y = 0.f;
    }
  }
}

// ---------------------------------------------------------------- coupling block B (Appendix A)
//
// B_SS' = 2 Bx_SS' - Bd_SS' couples the e-h pair S = (k, v, c) with the h-e pair (k', c' -> v'):
//   Bx_SS' = (1/(Omega Nk)) sum_{G != 0} conj(rho_vc^{kk}(G)) vbar(G) conj(rho_v'c'^{k'k'}(-G))
//   Bd_SS' = (1/(Omega Nk)) sum_{G,G'} conj(rho_vc'^{kk'}(G)) W_GG'(q) rho_cv'^{kk'}(G')
// B is symmetric: the upper blocks k <= k' are built and mirrored as B_k'k = B_kk'^T.

// rhot[S][G] = conj(rho_x[S][-G]) on the q = 0 sphere (the h-e pair density).
__global__ void minus_g_kernel(DevSys d, const float2* __restrict__ rho_x, float2* __restrict__ rhot) {
  const long long n = (long long)d.dim * d.ng0;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const int S = (int)(i / d.ng0), t = (int)(i - (long long)S * d.ng0);
    const int m = d.gminus0[t];
    const float2 v = m >= 0 ? rho_x[(size_t)S * d.ng_max + m] : make_float2(0.f, 0.f);
    rhot[(size_t)S * d.ng_max + t] = make_float2(v.x, -v.y);
  }
}

// B = 2 Bx on tiles touching k(S) <= k(S') (the exchange scale sqrt(2 vbar/(Omega Nk)) on both operands).
__global__ __launch_bounds__(kGemmThreads) void cpl_init_kernel(DevSys d, const float2* __restrict__ rho_x,
                                                                const float2* __restrict__ rhot,
                                                                float2* __restrict__ Bm) {
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  if (m0 >= d.dim || n0 >= d.dim) return;
  if (kpt_of_pair(d, m0) > kpt_of_pair(d, min(n0 + BN, d.dim) - 1)) return;
  __shared__ gemm::Smem sm;
  float2 acc[4][4];
  gemm::tile<true, true, true, false, true>(rho_x, d.ng_max, d.dim, rhot, d.ng_max, d.dim, d.ng0, m0, n0, sm, acc,
                                            d.xscale);
  const int tm = threadIdx.x / 16, tn = threadIdx.x % 16;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int S = m0 + tm * 4 + i;
    if (S >= d.dim) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int S2 = n0 + tn * 4 + j;
      if (S2 < d.dim) Bm[(size_t)S * d.dim + S2] = acc[i][j];
    }
  }
}

// Per upper block: M[a][c] = sum_G conj(Lv[a][G]) X[c][G], a = (v, c'), c = (c, v'), X = W rho_cv';
// B[(k,v,c)][(k',v',c')] -= M/(Omega Nk), mirror B_k'k = B_kk'^T, diagonal blocks (B + B^T)/2.
__global__ __launch_bounds__(kBlkThreads) void cpl_block_kernel(DevSys d, const float2* __restrict__ rho_cpl,
                                                               const float2* __restrict__ X, float2* __restrict__ Bm,
                                                               int q_begin, long long vbase) {
  __shared__ float2 Ls[16][KC + 1];
  __shared__ float2 Rs[16][KC + 1];
  __shared__ float2 Bs[16][17];
  const long long b0 = d.qblk_off[q_begin];
  const long long b = b0 + blockIdx.x;
  const int4 blk = d.blocks[b];
  const int k = blk.x, k2 = blk.y, q = blk.z;
  const long long qb = d.qblk_off[q];
  const long long local = b - qb;
  const int nv = d.nv, nc = d.nc, w = nv * nc;
  const float2* L = rho_cpl + (size_t)(2LL * w * qb - vbase + local * w) * d.ng_max;
  const float2* R = X + (size_t)((qb - b0 + local) * w) * d.ng_max;
  const int NG = d.ngq[q];
  const int t = threadIdx.x;
  const int a = t / w, c = t % w;
  const bool active = t < w * w;
  float2 acc = make_float2(0.f, 0.f);
  for (int g0 = 0; g0 < NG; g0 += KC) {
    for (int i = t; i < 16 * KC; i += kBlkThreads) {
      const int r = i / KC, g = i % KC;
      const bool in = r < w && (g0 + g) < NG;
      Ls[r][g] = in ? L[(size_t)r * d.ng_max + g0 + g] : make_float2(0.f, 0.f);
      Rs[r][g] = in ? R[(size_t)r * d.ng_max + g0 + g] : make_float2(0.f, 0.f);
    }
    __syncthreads();
    if (active) {
#pragma unroll 8
      for (int g = 0; g < KC; ++g) {
        const float2 l = Ls[a][g], r = Rs[c][g];
        acc.x = fmaf(l.x, r.x, fmaf(l.y, r.y, acc.x));     // conj(l) r
        acc.y = fmaf(l.x, r.y, fmaf(-l.y, r.x, acc.y));
      }
    }
    __syncthreads();
  }
  const float nrm = (float)d.norm;
  int row = 0, col = 0;
  float2 val = make_float2(0.f, 0.f);
  if (active) {
    const int v = a / nc, cp = a % nc, cc = c / nv, vp = c % nv;
    row = v * nc + cc;                 // (k, v, c) local
    col = vp * nc + cp;                // (k', v', c') local
    const size_t bij = (size_t)(k * w + row) * d.dim + (size_t)k2 * w + col;
    const float2 h = Bm[bij];
    val = make_float2(h.x - nrm * acc.x, h.y - nrm * acc.y);
    if (k != k2) {
      Bm[bij] = val;
      Bm[(size_t)(k2 * w + col) * d.dim + (size_t)k * w + row] = val;
    } else {
      Bs[row][col] = val;
    }
  }
  if (k == k2) {
    __syncthreads();
    if (active) {
      const float2 o = Bs[col][row];
      Bm[(size_t)(k * w + row) * d.dim + (size_t)k * w + col] = make_float2(0.5f * (val.x + o.x), 0.5f * (val.y + o.y));
    }
  }
}

// Lower blocks B_k'k = B_kk'^T and diagonal blocks (B + B^T)/2 for a build without the direct term.
__global__ void cpl_mirror_kernel(DevSys d, float2* __restrict__ Bm) {
  const long long n = (long long)d.dim * d.dim;
  const int nvc = d.nv * d.nc;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const int S = (int)(i / d.dim), S2 = (int)(i - (long long)S * d.dim);
    const int k = S / nvc, k2 = S2 / nvc;
    if (k > k2) {
      Bm[i] = Bm[(size_t)S2 * d.dim + S];
    } else if (k == k2 && S < S2) {
      const float2 a = Bm[i], b = Bm[(size_t)S2 * d.dim + S];
      const float2 m = make_float2(0.5f * (a.x + b.x), 0.5f * (a.y + b.y));
      Bm[i] = m;
      Bm[(size_t)S2 * d.dim + S] = m;
    }
  }
}

// k-point symmetry: block (ik, ik2) = representative block (or its conjugate transpose), and the mirror
// H_{ik2, ik} = H_{ik, ik2}^H; one CTA per listed block, one thread per element.
__global__ void symfill_kernel(DevSys d, float2* __restrict__ H) {
  const int4 f = d.fill[blockIdx.x];
  const int nvc = d.nv * d.nc;
  const bool mirrored = f.w < 0;
  const int ra = f.z, rb = mirrored ? -f.w - 1 : f.w;
  for (int t = threadIdx.x; t < nvc * nvc; t += blockDim.x) {
    const int i = t / nvc, j = t - i * nvc;
    float2 v;
    if (mirrored) {
      const float2 u = H[(size_t)(ra * nvc + j) * d.dim + rb * nvc + i];
      v = make_float2(u.x, -u.y);
    } else {
      v = H[(size_t)(ra * nvc + i) * d.dim + rb * nvc + j];
    }
    H[(size_t)(f.x * nvc + i) * d.dim + f.y * nvc + j] = v;
    if (f.x != f.y) H[(size_t)(f.y * nvc + j) * d.dim + f.x * nvc + i] = make_float2(v.x, -v.y);
  }
}
}  // namespace

int launch_symfill(const DevSys& d, void* H, void* stream) {
  if (d.nfill <= 0) return 0;
  if (d.nfill >= (1LL << 31)) return (int)cudaErrorInvalidValue;
  const int nvc = d.nv * d.nc;
  symfill_kernel<<<(unsigned)d.nfill, nvc * nvc < 256 ? (nvc * nvc + 31) / 32 * 32 : 256, 0, (cudaStream_t)stream>>>(
      d, (float2*)H);
  return (int)cudaGetLastError();
}

int launch_mirror(const DevSys& d, void* H, void* stream) {
  mirror_kernel<<<1216, 256, 0, (cudaStream_t)stream>>>(d, (float2*)H);
  return (int)cudaGetLastError();
}

// FP32 W.rho rows of a q chunk (w rows per block), followed by the split tile images of the products.
static size_t x_bytes(const DevSys& d, long long qchunk, long long w) {
  long long nb = qchunk * d.nkpt;
  if (nb > d.nblocks) nb = d.nblocks;
  return (((size_t)(nb * w) * d.ng_max * sizeof(float2)) + 255) & ~(size_t)255;
}

static long long direct_width(const DevSys& d) {
  return (d.nv * d.nv <= d.nc * d.nc) ? d.nv * d.nv : d.nc * d.nc;
}

// Split operand images of the W.rho products, in either precision.
static size_t split_bytes(const DevSys& d, long long qchunk, long long w) {
  const size_t a = tc_split_bytes(d, qchunk, w), b = wr32_split_bytes(d, qchunk, w);
  return a > b ? a : b;
}

// The direct stage's W.rho rows and split images of a q chunk; at least the exchange stage's split images of
// rho_x (BSE_BK_INIT).
size_t kernel_ws_bytes(const DevSys& d, long long qchunk) {
  const long long w = direct_width(d);
  const size_t direct = x_bytes(d, qchunk, w) + split_bytes(d, qchunk, w);
  const size_t init = gram32_ws_bytes(d) > gram_ws_bytes(d) ? gram32_ws_bytes(d) : gram_ws_bytes(d);
  return direct > init ? direct : init;
}

// Coupling build: W.rho_cv' rows and split images of a q chunk, or (init) conj(rho_x(-G)) rows.
size_t coupling_ws_bytes(const DevSys& d, long long qchunk) {
  const long long w = (long long)d.nv * d.nc;
  const size_t direct = qchunk > 0 ? x_bytes(d, qchunk, w) + split_bytes(d, qchunk, w) : 0;
  const size_t init = (((size_t)d.dim * d.ng_max * sizeof(float2)) + 255) & ~(size_t)255;
  return direct > init ? direct : init;
}

int launch_kernel_init(const DevSys& d, const void* rho_x, const double* energies, double delta, void* H,
                       void* stream) {
  dim3 grid((d.dim + BN - 1) / BN, (d.dim + BM - 1) / BM);
  init_kernel<<<grid, kGemmThreads, 0, (cudaStream_t)stream>>>(d, (const float2*)rho_x, energies, delta, (float2*)H);
  return (int)cudaGetLastError();
}

int launch_kernel_direct_range(const DevSys& d, const void* rho_dir, int q_begin, int q_end, long long b_begin,
                               long long b_count, long long vbase, long long max_rows, const void* W, int prec,
                               void* H, void* ws, int* status, void* stream) {
  const int side_c = (d.nc * d.nc < d.nv * d.nv) ? 1 : 0;
  cudaStream_t st = (cudaStream_t)stream;
  int e;
  if (prec != BSE_PREC_BF16X3 && prec != BSE_PREC_FP32) return -1;
  if (b_count <= 0 || max_rows <= 0) return 0;     // no block in the range (k-point symmetry can leave q empty)
  if (prec == BSE_PREC_BF16X3) {
    void* split_ws = (char*)ws + x_bytes(d, q_end - q_begin, direct_width(d));
    e = launch_gemm_wr_tc(d, rho_dir, q_begin, q_end, vbase, max_rows, W, ws, split_ws, side_c, status, stream);
  } else if (prec == BSE_PREC_FP32) {
    void* split_ws = (char*)ws + x_bytes(d, q_end - q_begin, direct_width(d));
    e = launch_gemm_wr(d, rho_dir, q_begin, q_end, vbase, max_rows, W, ws, split_ws, side_c, status, stream);
  } else {
    return -1;
  }
  if (e) return e;
  return launch_blocks(d, (const float2*)rho_dir, (const float2*)ws, (float2*)H, q_begin, vbase, side_c, b_count, st);
}

int launch_coupling_init(const DevSys& d, const void* rho_x, void* Bm, void* ws, void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  minus_g_kernel<<<1216, 256, 0, st>>>(d, (const float2*)rho_x, (float2*)ws);
  dim3 grid((d.dim + BN - 1) / BN, (d.dim + BM - 1) / BM);
  cpl_init_kernel<<<grid, kGemmThreads, 0, st>>>(d, (const float2*)rho_x, (const float2*)ws, (float2*)Bm);
  return (int)cudaGetLastError();
}

int launch_coupling_mirror(const DevSys& d, void* Bm, void* stream) {
  cpl_mirror_kernel<<<1216, 256, 0, (cudaStream_t)stream>>>(d, (float2*)Bm);
  return (int)cudaGetLastError();
}

int launch_coupling_direct_range(const DevSys& d, const void* rho_cpl, int q_begin, int q_end, long long b_count,
                                 long long vbase, long long max_rows, const void* W, int prec, void* Bm, void* ws,
                                 int* status, void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  const long long w = (long long)d.nv * d.nc;
  int e;
  if (prec == BSE_PREC_BF16X3) {
    void* split_ws = (char*)ws + x_bytes(d, q_end - q_begin, w);
    e = launch_gemm_wr_tc(d, rho_cpl, q_begin, q_end, vbase, max_rows, W, ws, split_ws, 2, status, stream);
  } else if (prec == BSE_PREC_FP32) {
    void* split_ws = (char*)ws + x_bytes(d, q_end - q_begin, w);
    e = launch_gemm_wr(d, rho_cpl, q_begin, q_end, vbase, max_rows, W, ws, split_ws, 2, status, stream);
  } else {
    return -1;
  }
  if (e) return e;
  if (b_count > 0)
    cpl_block_kernel<<<(unsigned)b_count, kBlkThreads, 0, st>>>(d, (const float2*)rho_cpl, (const float2*)ws,
                                                                (float2*)Bm, q_begin, vbase);
  return (int)cudaGetLastError();
}

}  // namespace bse
