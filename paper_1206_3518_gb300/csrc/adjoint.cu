// Adjoint of a spectral loss (step A9).
//
// eps_2(w) = -C Im[P^H R(z) P], R(z) = (z - H)^{-1}, z = w + i eta (Eq. epsilon_chi_bar in
// the TDA, Appendix A resolvent).  For g(w) = dL/deps_2(w) and any perturbation dH,
// dL = Re sum_ij conj(G_ij) dH_ij with G = -C sum_w g(w) i xt(w) x(w)^H, x = R(z)P,
// xt = R(conj z)P.  The Lanczos basis V (rows v_j) is recomputed, H V^T ~ V^T T, and
// R(z)P ~ |P| V^T y(z) with y(z) = (z - T)^{-1} e_0, so xt = |P| V^T conj(y).  The
// Hermitian part of G, the gradient for Hermitian perturbations of H, is then
//   G_h = V^T M_h conj(V),  M_h[j][l] = -C |P|^2 sum_w g(w) Im(y_j(w) y_l(w))   (real symmetric),
// and dL/dDelta = Re tr G = tr M_h (orthonormal basis).  y(z) is obtained stably from the
// tail continued fractions t_j = 1/(z - a_j - b_{j+1}^2 t_{j+1}): y_0 = t_0, y_j = b_j t_j y_{j-1}.
//
// Chain to the kernel inputs (H = diag + 2K^x - K^d, upper blocks k <= k' mirrored; the
// effective gradient of an upper block is 2 G_h for k < k' and G_h for k = k'):
//   dL/drho_x[S][G]   = 4 vbar(G)/(Omega Nk) sum_S' G_h[S'][S] rho_x[S'][G]
//   per upper block, Gm[vv'][cc'] = block gradient at ((k,v,c),(k',v',c')):
//   dL/drho_cc'[cc'] = -(1/(Omega Nk)) sum_vv' Gm[vv'][cc'] (W rho_vv')
//   dL/drho_vv'[vv'] = -(1/(Omega Nk)) sum_cc' conj(Gm[vv'][cc']) (W rho_cc')
//   dL/dW_q          = -(1/(Omega Nk)) sum_blocks sum_cc' Y[cc'] rho_cc'^H,  Y[cc'] = sum_vv' Gm rho_vv'
// every stored entry of rho and W taken as a free variable.
#include <cuda_runtime.h>

#include <algorithm>

#include "gemm_tile.cuh"
#include "internal.h"
#include "tcfcols.cuh"

namespace bse {
namespace {

constexpr int kNwChunk = 256;       // frequencies per resolvent chunk
constexpr int kQChunk = 32;         // q points per direct-term chunk

size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

size_t split_area(const DevSys& d, long long nsteps, long long qc);

struct BwdLayout {
  size_t spec, eps2, ab, done, scal, Y, Mh, Mf, Vf, Zf, Gh, Xv, Xc, Yd, split, total;
  long long rows_v, rows_c;
};

BwdLayout bwd_layout(const DevSys& d, long long nsteps) {
  BwdLayout L;
  const long long qc = kQChunk < d.nq ? kQChunk : d.nq;
  long long nb = qc * d.nkpt;
  if (nb > d.nblocks) nb = d.nblocks;
  L.rows_v = nb * d.nv * d.nv;
  L.rows_c = nb * d.nc * d.nc;
  size_t o = 0;
  L.spec = o; o = a256(o + spectrum_ws_bytes(d, nsteps));
  L.eps2 = o; o = a256(o + 8 * (size_t)kNwChunk);
  L.ab = o; o = a256(o + 16 * (size_t)nsteps);
  L.done = o; o = a256(o + 16);
  L.scal = o; o = a256(o + 64);
  L.Y = o; o = a256(o + 16 * (size_t)kNwChunk * nsteps);
  L.Mh = o; o = a256(o + 8 * (size_t)nsteps * nsteps);
  L.Mf = o; o = a256(o + 8 * (size_t)nsteps * nsteps);
  L.Vf = o; o = a256(o + 8 * (size_t)nsteps * d.dim);
  L.Zf = o; o = a256(o + 8 * (size_t)nsteps * d.dim);
  L.Gh = o; o = a256(o + 8 * (size_t)d.dim * d.dim);
  L.Xv = o; o = a256(o + 8 * (size_t)L.rows_v * d.ng_max);
  L.Xc = o; o = a256(o + 8 * (size_t)L.rows_c * d.ng_max);
  L.Yd = o; o = a256(o + 8 * (size_t)L.rows_c * d.ng_max);
  L.split = o; o = a256(o + split_area(d, nsteps, qc));
  L.total = o;
  return L;
}

__global__ void norm2_kernel(const double2* __restrict__ P, int n, double* out) {
  __shared__ double red[32];
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) s += P[i].x * P[i].x + P[i].y * P[i].y;
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    out[0] = t;
  }
}

// y(w) = (z - T)^{-1} e_0 for the frequencies of one chunk; Y[w][j], j < n.
__global__ void resolvent_kernel(const double* __restrict__ ab, int nsteps, const int* __restrict__ done,
                                 const double* __restrict__ omega, int w0, int nwc, double eta,
                                 double2* __restrict__ Y) {
  const int wi = blockIdx.x * blockDim.x + threadIdx.x;
  if (wi >= nwc) return;
  const int n = *done;
  const double zr = omega[w0 + wi], zi = eta;
  double2* y = Y + (size_t)wi * nsteps;
  double tr = 0.0, ti = 0.0;
  for (int j = n - 1; j >= 0; --j) {                 // tail fractions t_j
    double dr = zr - ab[j], di = zi;
    if (j + 1 < n) {
      const double b2 = ab[nsteps + j + 1] * ab[nsteps + j + 1];
      dr -= b2 * tr;
      di -= b2 * ti;
    }
    const double den = dr * dr + di * di;
    tr = dr / den;
    ti = -di / den;
    y[j] = make_double2(tr, ti);
  }
  double2 prev = y[0];                                // y_0 = t_0
  for (int j = 1; j < n; ++j) {
    const double b = ab[nsteps + j];
    const double2 t = y[j];
    const double2 cur = make_double2(b * (t.x * prev.x - t.y * prev.y), b * (t.x * prev.y + t.y * prev.x));
    y[j] = cur;
    prev = cur;
  }
}

// Mh[j][l] += -C |P|^2 sum_{w in chunk} g(w) Im(y_j y_l)  (j <= l, mirrored).
__global__ void mh_kernel(const double2* __restrict__ Y, int nsteps, const int* __restrict__ done,
                          const double* __restrict__ g, int w0, int nwc, const double* __restrict__ scal, double cpref,
                          double* __restrict__ Mh) {
  const int n = *done;
  const int j = blockIdx.y * 16 + threadIdx.y, l = blockIdx.x * 16 + threadIdx.x;
  if (j >= n || l >= n || j > l) return;
  double s = 0.0;
  for (int w = 0; w < nwc; ++w) {
    const double2 a = Y[(size_t)w * nsteps + j], b = Y[(size_t)w * nsteps + l];
    s += g[w0 + w] * (a.x * b.y + a.y * b.x);
  }
  const double v = -cpref * scal[0] * s;
  Mh[(size_t)j * nsteps + l] += v;
  if (j != l) Mh[(size_t)l * nsteps + j] += v;
}

// dL/dDelta = tr Mh; Mf = (complex64) Mh; Vf = (complex64) V.
__global__ void finish_m_kernel(const double* __restrict__ Mh, int nsteps, const int* __restrict__ done,
                                double* __restrict__ d_delta, float2* __restrict__ Mf) {
  const int n = *done;
  __shared__ double red[32];
  double s = 0.0;
  for (int j = threadIdx.x; j < n; j += blockDim.x) s += Mh[(size_t)j * nsteps + j];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  for (int i = threadIdx.x; i < nsteps * nsteps; i += blockDim.x) {
    const int j = i / nsteps, l = i % nsteps;
    Mf[i] = make_float2((j < n && l < n) ? (float)Mh[i] : 0.f, 0.f);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    *d_delta = t;
  }
}

// Vf = FP32 basis (the hi parts of the double-float split), zero beyond the steps done.
__global__ void v_to_float_kernel(const float4* __restrict__ V, long long n, const int* __restrict__ done, int dim,
                                  float2* __restrict__ Vf) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int j = (int)(i / dim);
  const float4 v = V[i];
  Vf[i] = (j < *done) ? make_float2(v.x + v.y, v.z + v.w) : make_float2(0.f, 0.f);
}

// Generic grouped product C = opA(A) opB(B)^T with per-column epilogue scale (dense, one group).
template <bool A_KC, bool B_KC, bool CA, bool CB>
__global__ __launch_bounds__(gemm::kThreads) void gemm_kernel(const float2* __restrict__ A, long long lda, int M,
                                                             const float2* __restrict__ B, long long ldb, int N, int K,
                                                             float2* __restrict__ C, long long ldc, float alpha,
                                                             const float* __restrict__ colscale2) {
  const int m0 = blockIdx.y * gemm::BM, n0 = blockIdx.x * gemm::BN;
  if (m0 >= M || n0 >= N) return;
  __shared__ gemm::Smem sm;
  float2 acc[4][4];
  gemm::tile<A_KC, B_KC, CA, CB>(A, lda, M, B, ldb, N, K, m0, n0, sm, acc);
  const int tm = threadIdx.x / 16, tn = threadIdx.x % 16;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = m0 + tm * 4 + i;
    if (r >= M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int c = n0 + tn * 4 + j;
      if (c >= N) continue;
      float sc = alpha;
      if (colscale2) sc *= colscale2[c] * colscale2[c];
      C[(size_t)r * ldc + c] = make_float2(sc * acc[i][j].x, sc * acc[i][j].y);
    }
  }
}

// Per upper block of the chunk: block gradient Gm, dL/drho_vv', dL/drho_cc' and Y = Gm-weighted rho_vv'.
__global__ __launch_bounds__(256) void block_grad_kernel(DevSys d, const float2* __restrict__ Gh,
                                                         const float2* __restrict__ rho_dir,
                                                         const float2* __restrict__ Xv, const float2* __restrict__ Xc,
                                                         float2* __restrict__ drho_dir, float2* __restrict__ Yd,
                                                         int q_begin) {
  __shared__ float2 Gm[16][16];
  const long long b0 = d.qblk_off[q_begin];
  const long long b = b0 + blockIdx.x;
  const int4 blk = d.blocks[b];
  const int k = blk.x, k2 = blk.y, q = blk.z;
  const long long qb = d.qblk_off[q];
  const long long nblk = d.qblk_off[q + 1] - qb;
  const long long local = b - qb;
  const int nv = d.nv, nc = d.nc, nv2 = nv * nv, nc2 = nc * nc, nvc = nv * nc;
  const float fac = (k == k2) ? 1.f : 2.f;
  for (int t = threadIdx.x; t < nv2 * nc2; t += blockDim.x) {
    const int a = t / nc2, c = t % nc2;
    const int v = a / nv, vp = a % nv, cc = c / nc, cp = c % nc;
    const float2 g = Gh[(size_t)(k * nvc + v * nc + cc) * d.dim + (size_t)k2 * nvc + vp * nc + cp];
    Gm[a][c] = make_float2(fac * g.x, fac * g.y);
  }
  __syncthreads();
  const long long vq = d.qvec_off[q];
  const float2* Rv = rho_dir + (size_t)(vq + local * nv2) * d.ng_max;
  float2* dRv = drho_dir ? drho_dir + (size_t)(vq + local * nv2) * d.ng_max : nullptr;
  float2* dRc = drho_dir ? drho_dir + (size_t)(vq + nblk * nv2 + local * nc2) * d.ng_max : nullptr;
  const float2* xv = Xv + (size_t)((qb - b0 + local) * nv2) * d.ng_max;
  const float2* xc = Xc + (size_t)((qb - b0 + local) * nc2) * d.ng_max;
  float2* y = Yd + (size_t)((qb - b0 + local) * nc2) * d.ng_max;
  const int NG = d.ngq[q];
  const float nrm = (float)d.norm;
  for (int G = threadIdx.x; G < NG; G += blockDim.x) {
    float2 rv[16], xvv[16], xcc[16];
    for (int a = 0; a < nv2; ++a) {
      rv[a] = Rv[(size_t)a * d.ng_max + G];
      xvv[a] = xv[(size_t)a * d.ng_max + G];
    }
    for (int c = 0; c < nc2; ++c) xcc[c] = xc[(size_t)c * d.ng_max + G];
    for (int c = 0; c < nc2; ++c) {
      float2 s1 = make_float2(0.f, 0.f), s2 = make_float2(0.f, 0.f);
      for (int a = 0; a < nv2; ++a) {
        const float2 g = Gm[a][c];
        s1.x += g.x * xvv[a].x - g.y * xvv[a].y;
        s1.y += g.x * xvv[a].y + g.y * xvv[a].x;
        s2.x += g.x * rv[a].x - g.y * rv[a].y;
        s2.y += g.x * rv[a].y + g.y * rv[a].x;
      }
      if (dRc) dRc[(size_t)c * d.ng_max + G] = make_float2(-nrm * s1.x, -nrm * s1.y);
      y[(size_t)c * d.ng_max + G] = s2;
    }
    if (dRv) {
      for (int a = 0; a < nv2; ++a) {
        float2 s = make_float2(0.f, 0.f);
        for (int c = 0; c < nc2; ++c) {
          const float2 g = Gm[a][c];            // conj(g) * xc
          s.x += g.x * xcc[c].x + g.y * xcc[c].y;
          s.y += g.x * xcc[c].y - g.y * xcc[c].x;
        }
        dRv[(size_t)a * d.ng_max + G] = make_float2(-nrm * s.x, -nrm * s.y);
      }
    }
  }
}

// ---------------------------------------------------------------- products on the tensor cores (tcf16.cuh)
//
// Measured, fcc 8x8x8 3v4c, 300 steps (64 x 64 tiles on the FP32 pipes before): dL/dW 43.0 -> 9.8 ms (products 4.8,
// images 5.0), dL/drho_x 3.1 -> 0.6, G_h 2.0 -> 0.3; error of dL/dW against 64 bits 2.7e-6 -> 2.0e-6 (what is left is
// the recursion's FP32 product).

// Columns of a dense operand X[k][g].
struct DenseSrc {
  const float2* x;
  int ld, K, G, nbatch;
  __device__ __forceinline__ bool get(int, const float2*& p, int& k, int& g) const {
    p = x;
    k = K;
    g = G;
    return true;
  }
};

// C[m][n] = alpha s(n)^2 sum_k opA(A[m][k]) B[n][k] of one pair of images; rows from m_begin (a panel of A).
template <bool CONJ>
struct DenseOp {
  static constexpr bool kReal = false, kConj = CONJ, kHerm = false;
  const unsigned char *a, *b;
  const float *inva, *invb;
  float2* C;
  int M, N, K, nt, n_tile, kc;
  long long ldc;
  float alpha;
  const float* colscale;
  int* status;
  long long ntiles;
  __device__ __forceinline__ bool tile(long long ti, tcf::Tile& o) const {
    const int mt = (int)(ti / nt), ntl = (int)(ti - (long long)mt * nt);
    o.a_step = 2 * tcf::kTileA;
    o.b_step = (uint32_t)(2 * n_tile * umma::kRow);
    o.a = a + (size_t)mt * kc * o.a_step;
    o.b = b + (size_t)ntl * kc * o.b_step;
    o.K = K;
    o.n = n_tile;
    o.m0 = mt * tcf::kTM;
    o.n0 = ntl * n_tile;
    o.mvalid = M - o.m0;
    o.nvalid = min(n_tile, N - o.n0);
    o.batch = 0;
    o.row0 = o.m0;
    return true;
  }
  __device__ __forceinline__ float2* row_out(const tcf::Tile& t, int row) const { return C + (t.row0 + row) * ldc + t.n0; }
  __device__ __forceinline__ float row_scale(const tcf::Tile& t, int row) const { return inva[t.m0 + row]; }
  __device__ __forceinline__ float col_scale(const tcf::Tile& t, int col) const { return invb[t.n0 + col]; }
  __device__ __forceinline__ float2 value(const tcf::Tile& t, int, int col, float2 v) const {
    float s = alpha;
    if (colscale) s *= colscale[t.n0 + col] * colscale[t.n0 + col];
    return make_float2(s * v.x, s * v.y);
  }
};

// Columns of the rows of one band side of a q chunk: rho_cc' (rho_dir) or Y (its chunk).
struct SideSrc {
  DevSys d;
  const float2* x;
  int q_begin, ld, nbatch;
  bool chunk;                                   // x starts at the chunk's first block, rows of Nc^2 only
  __device__ __forceinline__ bool get(int batch, const float2*& p, int& K, int& G) const {
    const int q = q_begin + batch, nc2 = d.nc * d.nc;
    const long long nblk = d.qblk_off[q + 1] - d.qblk_off[q];
    const long long row = chunk ? (d.qblk_off[q] - d.qblk_off[q_begin]) * nc2 : d.qvec_off[q] + nblk * d.nv * d.nv;
    p = x + (size_t)row * d.ng_max;
    K = (int)(nblk * nc2);
    G = d.ngq[q];
    return K > 0;
  }
};

// dW_q[G][G'] = -norm sum_k Y_q[k][G] conj(Rc_q[k][G']) over the q chunk, as -norm conj(conj(Y)^T Rc).
struct DwOp {
  static constexpr bool kReal = false, kConj = true, kHerm = false;
  DevSys d;
  const unsigned char *a, *b;
  const float *inva, *invb;
  float2* dW;
  size_t a_batch, b_batch;
  int q_begin, mt, nt, n_tile, kc;
  int* status;
  long long ntiles;
  __device__ __forceinline__ bool tile(long long ti, tcf::Tile& o) const {
    const int ntl = (int)(ti % nt);
    const long long r = ti / nt;
    const int mtl = (int)(r % mt), qi = (int)(r / mt), q = q_begin + qi, NG = d.ngq[q];
    o.m0 = mtl * tcf::kTM;
    o.n0 = ntl * n_tile;
    o.K = (int)(d.qblk_off[q + 1] - d.qblk_off[q]) * d.nc * d.nc;
    if (o.m0 >= NG || o.n0 >= NG || o.K == 0) return false;
    o.a_step = 2 * tcf::kTileA;
    o.b_step = (uint32_t)(2 * n_tile * umma::kRow);
    o.a = a + qi * a_batch + (size_t)mtl * kc * o.a_step;
    o.b = b + qi * b_batch + (size_t)ntl * kc * o.b_step;
    o.n = n_tile;
    o.mvalid = NG - o.m0;
    o.nvalid = min(n_tile, NG - o.n0);
    o.batch = qi;
    o.row0 = (long long)q * d.ng_max + o.m0;
    return true;
  }
  __device__ __forceinline__ float2* row_out(const tcf::Tile& t, int row) const {
    return dW + (size_t)(t.row0 + row) * d.ng_max + t.n0;
  }
  __device__ __forceinline__ float row_scale(const tcf::Tile& t, int row) const {
    return inva[(size_t)t.batch * d.ng_max + t.m0 + row];
  }
  __device__ __forceinline__ float col_scale(const tcf::Tile& t, int col) const {
    return invb[(size_t)t.batch * d.ng_max + t.n0 + col];
  }
  __device__ __forceinline__ float2 value(const tcf::Tile&, int, int, float2 v) const {
    const float nrm = (float)d.norm;
    return make_float2(-nrm * v.x, nrm * v.y);
  }
};

// Rows of G_h (a panel): image rows, K = dim.
__global__ __launch_bounds__(256) void split_rows_kernel(const float2* __restrict__ x, long long ld, int rows, int K,
                                                         unsigned char* __restrict__ img, float* __restrict__ inv,
                                                         int kc) {
  const int row = blockIdx.x * 8 + (threadIdx.x >> 5);
  const bool live = row < rows;
  const float s = tcf::split_row<32, 3>(x + (size_t)(live ? row : 0) * ld, K, nullptr,
                                        img + (size_t)(row / tcf::kTM) * kc * (2 * tcf::kTileA), 2 * tcf::kTileA,
                                        tcf::kTileA, row % tcf::kTM, live);
  if (live && (threadIdx.x & 31) == 0) inv[row] = s;
}

constexpr int kPanel = 32 * tcf::kTM;           // rows of G_h split at a time (the images of all would take its size again)

// q points of a chunk of qc whose images are held at a time: as many as fit in 1.5 GiB, in groups of one size.  (fcc 8x8x8
// 3v4c: whole chunks, dW 1.5 GB; with 1 GiB and dW in two groups the gradient took 57.4 instead of 56.7 ms.  fcc 12x12x12
// 4v4c: whole chunks would take 3.7 GB for W.rho and 8.5 GB for dW.)
constexpr size_t kSplitArea = size_t(3) << 29;
int split_group(size_t per_q, long long qc) {
  const long long parts = (long long)((per_q * qc + kSplitArea - 1) / kSplitArea);
  return (int)((qc + parts - 1) / parts);
}
long long wide_side(const DevSys& d) { return d.nv > d.nc ? d.nv * d.nv : d.nc * d.nc; }
int wr_group(const DevSys& d, long long qc) { return split_group(wr32_split_bytes(d, 1, wide_side(d)), qc); }
int dw_group(const DevSys& d, long long qc) {
  const int K = d.nkpt * d.nc * d.nc;
  return split_group(tcf::cols_batch_bytes(d.ng_max, K, tcf::kTM) + tcf::cols_batch_bytes(d.ng_max, K, tcf::n_tile(d.ng_max)), qc);
}

// Largest use of the split area (images, then inverse scales): W.rho and dW of a group of q, G_h, dL/drho_x.
size_t split_area(const DevSys& d, long long nsteps, long long qc) {
  const int n = tcf::n_tile(d.ng_max), nd = tcf::n_tile(d.dim), n0 = tcf::n_tile(d.ng0);
  const int K = d.nkpt * d.nc * d.nc;
  const size_t wr = wr32_split_bytes(d, wr_group(d, qc), wide_side(d)), g = dw_group(d, qc);
  const size_t dw = a256(g * tcf::cols_batch_bytes(d.ng_max, K, tcf::kTM)) + a256(g * tcf::cols_batch_bytes(d.ng_max, K, n)) +
                    2 * a256(g * d.ng_max * 4);
  const size_t gh = a256(tcf::cols_batch_bytes(d.dim, (int)nsteps, tcf::kTM)) +
                    a256(tcf::cols_batch_bytes(d.dim, (int)nsteps, nd)) + 2 * a256((size_t)d.dim * 4);
  const size_t dx = a256(tcf::cols_batch_bytes(d.dim < kPanel ? d.dim : kPanel, d.dim, tcf::kTM)) +
                    a256(tcf::cols_batch_bytes(d.ng0, d.dim, n0)) + a256((size_t)kPanel * 4) + a256((size_t)d.ng_max * 4);
  return std::max(std::max(wr, dw), std::max(gh, dx));
}

// dL/dW of a group of q from Y (its first row that of q0) and rho_cc'.
int launch_dw(const DevSys& d, const float2* Yd, const float2* rho_dir, float2* dW, int q0, int q1, long long maxb,
              char* area, int* status, cudaStream_t st) {
  const int nq = q1 - q0, n = tcf::n_tile(d.ng_max), K = (int)maxb * d.nc * d.nc;
  if (K <= 0) return 0;
  const size_t ab = tcf::cols_batch_bytes(d.ng_max, K, tcf::kTM), bb = tcf::cols_batch_bytes(d.ng_max, K, n);
  unsigned char* a = (unsigned char*)area;
  unsigned char* b = a + a256(nq * ab);
  float* inva = (float*)(b + a256(nq * bb));
  float* invb = (float*)((char*)inva + a256((size_t)nq * d.ng_max * 4));
  int e = tcf::split_cols(SideSrc{d, Yd, q0, d.ng_max, nq, true}, K, d.ng_max, inva, a, tcf::kTM, st);
  if (!e) e = tcf::split_cols(SideSrc{d, rho_dir, q0, d.ng_max, nq, false}, K, d.ng_max, invb, b, n, st);
  if (e) return e;
  DwOp op{d, a, b, inva, invb, dW, ab, bb, q0, (d.ng_max + tcf::kTM - 1) / tcf::kTM, (d.ng_max + n - 1) / n, n,
          (K + tcf::kTKC - 1) / tcf::kTKC, status, 0};
  op.ntiles = (long long)nq * op.mt * op.nt;
  return tcf::launch(op, st);
}

// G_h = V^T Z (dim x dim, K = nsteps).
int launch_gh(const DevSys& d, const float2* Vf, const float2* Zf, int nsteps, float2* Gh, char* area, int* status,
              cudaStream_t st) {
  const int n = tcf::n_tile(d.dim), kc = (nsteps + tcf::kTKC - 1) / tcf::kTKC;
  unsigned char* a = (unsigned char*)area;
  unsigned char* b = a + a256(tcf::cols_batch_bytes(d.dim, nsteps, tcf::kTM));
  float* inva = (float*)(b + a256(tcf::cols_batch_bytes(d.dim, nsteps, n)));
  float* invb = (float*)((char*)inva + a256((size_t)d.dim * 4));
  int e = tcf::split_cols(DenseSrc{Vf, d.dim, nsteps, d.dim, 1}, nsteps, d.dim, inva, a, tcf::kTM, st);
  if (!e) e = tcf::split_cols(DenseSrc{Zf, d.dim, nsteps, d.dim, 1}, nsteps, d.dim, invb, b, n, st);
  if (e) return e;
  DenseOp<false> op{a, b, inva, invb, Gh, d.dim, d.dim, nsteps, (d.dim + n - 1) / n, n, kc, d.dim, 1.f, nullptr, status, 0};
  op.ntiles = (long long)((d.dim + tcf::kTM - 1) / tcf::kTM) * op.nt;
  return tcf::launch(op, st);
}

// dL/drho_x[S][G] = 2 xscale(G)^2 sum_S' conj(G_h[S][S']) rho_x[S'][G], G_h split a panel of rows at a time.
int launch_drho_x(const DevSys& d, const float2* Gh, const float2* rho_x, float2* drho_x, char* area, int* status,
                  cudaStream_t st) {
  const int n = tcf::n_tile(d.ng0), kc = (d.dim + tcf::kTKC - 1) / tcf::kTKC;
  unsigned char* a = (unsigned char*)area;
  unsigned char* b = a + a256(tcf::cols_batch_bytes(d.dim < kPanel ? d.dim : kPanel, d.dim, tcf::kTM));
  float* inva = (float*)(b + a256(tcf::cols_batch_bytes(d.ng0, d.dim, n)));
  float* invb = (float*)((char*)inva + a256((size_t)kPanel * 4));
  int e = tcf::split_cols(DenseSrc{rho_x, d.ng_max, d.dim, d.ng0, 1}, d.dim, d.ng0, invb, b, n, st);
  for (int m = 0; m < d.dim && !e; m += kPanel) {
    const int rows = d.dim - m < kPanel ? d.dim - m : kPanel;
    split_rows_kernel<<<(rows + 7) / 8, 256, 0, st>>>(Gh + (size_t)m * d.dim, d.dim, rows, d.dim, a, inva, kc);
    if ((e = (int)cudaGetLastError())) break;
    DenseOp<true> op{a, b, inva, invb, drho_x + (size_t)m * d.ng_max, rows, d.ng0, d.dim, (d.ng0 + n - 1) / n, n, kc,
                     d.ng_max, 2.f, d.xscale, status, 0};
    op.ntiles = (long long)((rows + tcf::kTM - 1) / tcf::kTM) * op.nt;
    e = tcf::launch(op, st);
  }
  return e;
}

}  // namespace

size_t backward_ws_bytes(const DevSys& d, long long nsteps) { return bwd_layout(d, nsteps).total; }



int launch_backward(const DevSys& d, const long long* h_qblk_off, const long long* h_qvec_off, const void* H,
                    const void* P, int nsteps, const double* omega, int nw, double eta, const double* dL,
                    const void* rho_x, const void* rho_dir, const void* W, double* d_delta, void* dH, void* drho_x,
                    void* drho_dir, void* dW, void* ws, int* status, void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  const BwdLayout L = bwd_layout(d, nsteps);
  char* base = (char*)ws;
  double* ab = (double*)(base + L.ab);
  int* done = (int*)(base + L.done);
  double* scal = (double*)(base + L.scal);
  double2* Y = (double2*)(base + L.Y);
  double* Mh = (double*)(base + L.Mh);
  float2* Mf = (float2*)(base + L.Mf);
  float2* Vf = (float2*)(base + L.Vf);
  float2* Zf = (float2*)(base + L.Zf);
  float2* Gh = dH ? (float2*)dH : (float2*)(base + L.Gh);
  float4* V = nullptr;
  // 1. Lanczos recomputed (the spectrum it evaluates on the first frequencies is not used).
  int e = run_haydock(d, H, P, nsteps, omega, nw < kNwChunk ? nw : kNwChunk, eta, (double*)(base + L.eps2), ab, done,
                      base + L.spec, status, stream, &V);
  if (e) return e;
  norm2_kernel<<<1, 1024, 0, st>>>((const double2*)P, d.dim, scal);
  // 2. M_h from the Krylov resolvent, chunked over frequencies.
  if ((e = (int)cudaMemsetAsync(Mh, 0, 8 * (size_t)nsteps * nsteps, st))) return e;
  for (int w0 = 0; w0 < nw; w0 += kNwChunk) {
    const int nwc = (nw - w0) < kNwChunk ? (nw - w0) : kNwChunk;
    resolvent_kernel<<<(nwc + 127) / 128, 128, 0, st>>>(ab, nsteps, done, omega, w0, nwc, eta, Y);
    dim3 g16((nsteps + 15) / 16, (nsteps + 15) / 16);
    mh_kernel<<<g16, dim3(16, 16), 0, st>>>(Y, nsteps, done, dL, w0, nwc, scal, d.prefactor, Mh);
  }
  finish_m_kernel<<<1, 1024, 0, st>>>(Mh, nsteps, done, d_delta, Mf);
  const long long nv_el = (long long)nsteps * d.dim;
  v_to_float_kernel<<<(unsigned)((nv_el + 255) / 256), 256, 0, st>>>(V, nv_el, done, d.dim, Vf);
  if ((e = (int)cudaGetLastError())) return e;
  // 3. Z = M_h conj(V) (n x dim), G_h = V^T Z (dim x dim), FP32 products.
  {
    dim3 gz((d.dim + 63) / 64, (nsteps + 63) / 64);
    gemm_kernel<true, false, false, true><<<gz, gemm::kThreads, 0, st>>>(Mf, nsteps, nsteps, Vf, d.dim, d.dim, nsteps,
                                                                        Zf, d.dim, 1.f, nullptr);
    if ((e = (int)cudaGetLastError())) return e;
    if ((e = launch_gh(d, Vf, Zf, nsteps, Gh, base + L.split, status, st))) return e;
  }
  // 4. exchange: dL/drho_x[S][G] = 2 xscale(G)^2 sum_S' conj(G_h[S][S']) rho_x[S'][G]
  if (drho_x) {
    if ((e = (int)cudaMemsetAsync(drho_x, 0, 8 * (size_t)d.dim * d.ng_max, st))) return e;
    if ((e = launch_drho_x(d, Gh, (const float2*)rho_x, (float2*)drho_x, base + L.split, status, st))) return e;
  }
  // 5. direct term, q chunks
  if (drho_dir || dW) {
    if (drho_dir && (e = (int)cudaMemsetAsync(drho_dir, 0, 8 * (size_t)h_qvec_off[d.nq] * d.ng_max, st))) return e;
    if (dW && (e = (int)cudaMemsetAsync(dW, 0, 8 * (size_t)d.nq * d.ng_max * d.ng_max, st))) return e;
    float2* Xv = (float2*)(base + L.Xv);
    float2* Xc = (float2*)(base + L.Xc);
    float2* Yd = (float2*)(base + L.Yd);
    for (int q0 = 0; q0 < d.nq; q0 += kQChunk) {
      const int q1 = (q0 + kQChunk) < d.nq ? q0 + kQChunk : d.nq;
      long long maxb = 0;
      for (int q = q0; q < q1; ++q) maxb = std::max(maxb, h_qblk_off[q + 1] - h_qblk_off[q]);
      const int gw = wr_group(d, kQChunk < d.nq ? kQChunk : d.nq), gd = dw_group(d, kQChunk < d.nq ? kQChunk : d.nq);
      for (int side = 0; side < 2; ++side)
        for (int qa = q0; qa < q1; qa += gw) {
          const int qb = std::min(q1, qa + gw), w = side ? d.nc * d.nc : d.nv * d.nv;
          float2* X = (side ? Xc : Xv) + (size_t)((h_qblk_off[qa] - h_qblk_off[q0]) * w) * d.ng_max;
          if ((e = launch_gemm_wr(d, rho_dir, qa, qb, 0, maxb * w, W, X, base + L.split, side, status, stream))) return e;
        }
      const long long nb = h_qblk_off[q1] - h_qblk_off[q0];
      if (nb > 0)
        block_grad_kernel<<<(unsigned)nb, 256, 0, st>>>(d, Gh, (const float2*)rho_dir, Xv, Xc, (float2*)drho_dir, Yd,
                                                        q0);
      if ((e = (int)cudaGetLastError())) return e;
      for (int qa = q0; dW && qa < q1; qa += gd) {
        const float2* Y = Yd + (size_t)((h_qblk_off[qa] - h_qblk_off[q0]) * d.nc * d.nc) * d.ng_max;
        if ((e = launch_dw(d, Y, (const float2*)rho_dir, (float2*)dW, qa, std::min(q1, qa + gd), maxb, base + L.split, status,
                           st)))
          return e;
      }
    }
  }
  return 0;
}

}  // namespace bse
