// Static RPA screening from the system's own states (Sec. II A-B, Eqs. chi0_GG, epsilon_-1;
// the W_GG'(q) form of Sec. III A).  Not on the spectrum path: it produces the W that step A4
// otherwise takes as input.
//
//   a_S(G)  = sqrt(|w_S|) v^1/2(q+G) rho_vc^{k,k+q}(G),  w_S = 4/(Omega Nk)/(e_vk - e_c,k+q) < 0
//             (q = 0: a_S(0) = sqrt(|w_S|) sqrt(4 pi) conj(P_S), the k.p optical limit)
//   eps(q)  = I + sum_S a_S a_S^H            (= 1 - v^1/2 chi0 v^1/2, Hermitian, eigenvalues >= 1)
//   eps^-1  by Newton-Schulz: X <- X (2 I - eps X) from X_0 = 2/(1 + R) I, R a Gershgorin bound of
//           the largest eigenvalue, so |I - eps X_k| <= ((R - 1)/(R + 1))^(2^k)
//   W(q)    = v^1/2 eps^-1 v^1/2; at q = 0 the head is the mini-zone average [eps^-1]_00 12 pi/q_c^2
//             and the wings are zero.
//
// Everything is batched over the q points of a range.  The products are FP16x3 with promoted accumulation (tcf16.cuh,
// FP32 accuracy).  With X and eps Hermitian a step is T = 2 I - X eps, Y = X T^H (= 2 X - X eps X), so that every
// operand enters by its rows (sum_k A_mk conj(B_nk)); Y is computed on the upper triangle and mirrored, which keeps X
// exactly Hermitian (an anti-Hermitian part of X would double in each step).
//
// Measured, fcc 8x8x8 3v4c, 64 q, 16 steps: 4.8 ms beside the pair densities' 7.1 (Newton-Schulz products
// 2.2, eps 0.9, splits 0.9, scaling 0.6), error of W against 64 bits 1.8e-7; with 64 x 64 tiles on the FP32 pipes and the
// weights' FP64 roots taken per element 24.2 ms (13.2, 7.5, -, 3.2), 2.2e-6 to 3.2e-6.
#include <cuda_runtime.h>

#include <algorithm>

#include "internal.h"
#include "tcfcols.cuh"

namespace bse {
namespace {

using tcf::kTileA;
using tcf::kTKC;
using tcf::kTM;
constexpr size_t kImgBytes = size_t(1) << 30;     // images of pair vectors at a time,
constexpr int kQImg = 32;                        // of at most so many q points

// sw[row] = sqrt(|w_S|), row = ((qi Nk + k) Nv + v) Nc + c.
__global__ void weight_kernel(DevSys d, const double* __restrict__ e, int q_begin, long long rows, double gap_floor,
                              float* __restrict__ sw) {
  const long long row = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= rows) return;
  const int nvc = d.nv * d.nc;
  const int qi = (int)(row / ((long long)d.nkpt * nvc));
  const int rem = (int)(row - (long long)qi * d.nkpt * nvc);
  const int k = rem / nvc, iv = (rem / d.nc) % d.nv, ic = rem % d.nc;
  const int q = q_begin + qi;
  const int k1 = k / (d.nk2 * d.nk3), k2 = (k / d.nk3) % d.nk2, k3 = k % d.nk3;
  const int q1 = q / (d.nk2 * d.nk3), q2 = (q / d.nk3) % d.nk2, q3 = q % d.nk3;
  const int kp = (((k1 + q1) % d.nk1) * d.nk2 + (k2 + q2) % d.nk2) * d.nk3 + (k3 + q3) % d.nk3;
  const double de = fmax(e[(size_t)kp * d.nb + d.nv + ic] - e[(size_t)k * d.nb + iv], gap_floor);
  sw[row] = (float)sqrt(4.0 / (d.omega_cell * d.nkpt * de));
}

constexpr int kScaleRows = 64;

// In place: rho rows -> a rows (q-range layout [q][k][v][c][ng_max]), and the largest component of every column of a q
// (bits of the absolute value).  64 rows per CTA, a thread per column.
__global__ __launch_bounds__(256) void scale_kernel(DevSys d, float2* __restrict__ a, const float* __restrict__ sw,
                                                    const double2* __restrict__ P, int q_begin, int K,
                                                    unsigned* __restrict__ mx) {
  const int qi = blockIdx.y, q = q_begin + qi, r0 = blockIdx.x * kScaleRows;
  const int NG = d.ngq[q], nr = min(kScaleRows, K - r0);
  __shared__ float w[kScaleRows];
  const long long base = (long long)qi * K + r0;
  if (threadIdx.x < nr) w[threadIdx.x] = sw[base + threadIdx.x];
  __syncthreads();
  const float* vs = d.vsq + (size_t)q * d.ng_max;
  for (int g = threadIdx.x; g < d.ng_max; g += blockDim.x) {
    float2* x = a + (size_t)base * d.ng_max + g;
    const float v = vs[g];                        // zero past the sphere
    float m = 0.f;
    for (int i = 0; i < nr; ++i, x += d.ng_max) {
      float2 y = make_float2(0.f, 0.f);
      if (q == 0 && g == 0) {
        const double2 p = P[r0 + i];              // conj(P_S) sqrt(4 pi)
        const double f = 3.5449077018110320546 * (double)w[i];
        y = make_float2((float)(p.x * f), (float)(-p.y * f));
      } else if (g < NG) {
        const float2 r = *x;
        const float f = w[i] * v;
        y = make_float2(r.x * f, r.y * f);
      }
      *x = y;
      m = fmaxf(m, fmaxf(fabsf(y.x), fabsf(y.y)));
    }
    if (m > 0.f) atomicMax(mx + (size_t)qi * d.ng_max + g, __float_as_uint(m));
  }
}

// Columns of the a rows of q.
struct VecSrc {
  const int* ngq;
  const float2* a;
  int q_begin, K, ld, nbatch;
  __device__ __forceinline__ bool get(int batch, const float2*& p, int& k, int& g) const {
    p = a + (size_t)batch * K * ld;
    k = K;
    g = ngq[q_begin + batch];
    return true;
  }
};

struct QGeo {                                     // images of ng_max rows of a q: nt tiles of `tile` rows, kc chunks each
  int ng_max, tile, nt, kc;
  size_t batch;                                   // bytes per q
};
QGeo qgeo(const DevSys& d, int K, int tile) {
  QGeo g;
  g.ng_max = d.ng_max;
  g.tile = tile;
  g.nt = (d.ng_max + tile - 1) / tile;
  g.kc = (K + kTKC - 1) / kTKC;
  g.batch = (size_t)g.nt * g.kc * (2 * (size_t)tile * umma::kRow);
  return g;
}

int q_images(const DevSys& d) {
  const size_t n = kImgBytes / qgeo(d, d.nkpt * d.nv * d.nc, kTM).batch;
  return n < 1 ? 1 : (int)std::min<size_t>(n, kQImg);
}

// C_q = f(sum_k A_mk conj(B_nk)) over the q of a range.
// MODE 0: eps = I + v; 1: alpha I + beta v; 2: v, Hermitian (upper tiles, mirrored).
template <int MODE>
struct QOp {
  static constexpr bool kReal = false, kConj = true, kHerm = MODE == 2;
  const int* ngq;
  QGeo g, gb;                                     // images of A (128-row tiles) and of B
  const unsigned char *a, *b;
  const float *inva, *invb;
  float2* C;
  int q_begin, K;                                 // K = 0: the sphere of q
  float alpha, beta;
  int* status;
  long long ntiles;
  __device__ __forceinline__ bool tile(long long ti, tcf::Tile& o) const {
    const int per = g.nt * gb.nt, qi = (int)(ti / per), r = (int)(ti - (long long)qi * per);
    const int I = r / gb.nt, J = r - I * gb.nt, NG = ngq[q_begin + qi];
    o.m0 = I * kTM;
    o.n0 = J * gb.tile;
    if ((kHerm && o.m0 >= o.n0 + gb.tile) || o.m0 >= NG || o.n0 >= NG) return false;
    o.a_step = 2 * kTileA;
    o.b_step = (uint32_t)(2 * gb.tile * umma::kRow);
    o.a = a + qi * g.batch + (size_t)I * g.kc * o.a_step;
    o.b = b + qi * gb.batch + (size_t)J * gb.kc * o.b_step;
    o.K = K ? K : NG;
    o.n = gb.tile;
    o.nvalid = min(gb.tile, NG - o.n0);
    o.mvalid = NG - o.m0;
    o.batch = qi;
    o.row0 = o.m0;
    return true;
  }
  __device__ __forceinline__ float2* row_out(const tcf::Tile& t, int row) const {
    return C + ((size_t)t.batch * g.ng_max + t.m0 + row) * g.ng_max + t.n0;
  }
  __device__ __forceinline__ float2* mirror_out(const tcf::Tile& t, int row, int col) const {
    return C + ((size_t)t.batch * g.ng_max + t.n0 + col) * g.ng_max + t.m0 + row;
  }
  __device__ __forceinline__ float row_scale(const tcf::Tile& t, int row) const {
    return inva[(size_t)t.batch * g.ng_max + t.m0 + row];
  }
  __device__ __forceinline__ float col_scale(const tcf::Tile& t, int col) const {
    return invb[(size_t)t.batch * g.ng_max + t.n0 + col];
  }
  __device__ __forceinline__ float2 value(const tcf::Tile& t, int row, int col, float2 v) const {
    const bool diag = t.m0 + row == t.n0 + col;
    if (MODE == 2) return make_float2(v.x, -v.y);
    const float b = MODE == 0 ? 1.f : beta;
    return make_float2(b * v.x + (diag ? (MODE == 0 ? 1.f : alpha) : 0.f), -b * v.y);
  }
};

// Row images of an NG x NG matrix per q (row stride ng_max); blockIdx.y = q.
template <int GL, int NP>
__global__ __launch_bounds__(256) void split_matrix_kernel(DevSys d, QGeo g, const float2* __restrict__ A,
                                                           unsigned char* __restrict__ img, float* __restrict__ inv,
                                                           int q_begin) {
  const int qi = blockIdx.y, NG = d.ngq[q_begin + qi], row = blockIdx.x * (256 / GL) + threadIdx.x / GL;
  const bool live = row < NG;
  const size_t at = (size_t)qi * d.ng_max + (live ? row : 0);
  const uint32_t lo = (uint32_t)(g.tile * umma::kRow);
  const float s = tcf::split_row<GL, NP>(A + at * d.ng_max, NG, nullptr,
                                         img + qi * g.batch + (size_t)(row / g.tile) * g.kc * (2 * (size_t)lo),
                                         2 * (size_t)lo, lo, row % g.tile, live);
  if (live && threadIdx.x % GL == 0) inv[at] = s;
}

template <int GL, int NP>
void split_rows(const DevSys& d, const QGeo& g, const float2* A, unsigned char* img, float* inv, int q_begin, int nq,
                cudaStream_t st) {
  constexpr int rows = 256 / GL;
  split_matrix_kernel<GL, NP><<<dim3((d.ng_max + rows - 1) / rows, nq), 256, 0, st>>>(d, g, A, img, inv, q_begin);
}
int split_matrix(const DevSys& d, const QGeo& g, const float2* A, unsigned char* img, float* inv, int q_begin, int nq,
                 cudaStream_t st) {
  if (d.ng_max <= 128)
    split_rows<16, 1>(d, g, A, img, inv, q_begin, nq, st);
  else if (d.ng_max <= 384)
    split_rows<16, 3>(d, g, A, img, inv, q_begin, nq, st);
  else
    split_rows<32, 3>(d, g, A, img, inv, q_begin, nq, st);
  return (int)cudaGetLastError();
}

// R[q] = max row sum of |eps| (Gershgorin bound of the largest eigenvalue), as bits; one warp per row.
__global__ __launch_bounds__(256) void gershgorin_kernel(DevSys d, const float2* __restrict__ eps, unsigned* __restrict__ R,
                                                         int q_begin) {
  const int qi = blockIdx.y, NG = d.ngq[q_begin + qi], row = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (row >= NG) return;
  const float2* E = eps + ((size_t)qi * d.ng_max + row) * d.ng_max;
  float s = 0.f;
  for (int c = threadIdx.x & 31; c < NG; c += 32) {
    const float2 v = E[c];
    s += sqrtf(v.x * v.x + v.y * v.y);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) atomicMax(R + qi, __float_as_uint(s));
}

// X = 2/(1 + R) I.
__global__ void ns_init_kernel(DevSys d, const unsigned* __restrict__ R, float2* __restrict__ X, int q_begin) {
  const int qi = blockIdx.y, NG = d.ngq[q_begin + qi];
  const float x0 = 2.f / (1.f + __uint_as_float(R[qi]));
  float2* Xq = X + (size_t)qi * d.ng_max * d.ng_max;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < (long long)d.ng_max * d.ng_max;
       i += (long long)gridDim.x * blockDim.x) {
    const int r = (int)(i / d.ng_max), c = (int)(i % d.ng_max);
    Xq[i] = make_float2((r == c && r < NG) ? x0 : 0.f, 0.f);
  }
}

// residual[q] = max |I - eps X| (from T = eps X).
__global__ void residual_kernel(DevSys d, const float2* __restrict__ T, float* __restrict__ res, int q_begin) {
  const int qi = blockIdx.x, q = q_begin + qi;
  const int NG = d.ngq[q];
  const float2* Tq = T + (size_t)qi * d.ng_max * d.ng_max;
  float m = 0.f;
  for (long long i = threadIdx.x; i < (long long)NG * NG; i += blockDim.x) {
    const int r = (int)(i / NG), c = (int)(i % NG);
    float2 v = Tq[(size_t)r * d.ng_max + c];
    if (r == c) v.x -= 1.f;
    m = fmaxf(m, sqrtf(v.x * v.x + v.y * v.y));
  }
  __shared__ float red[32];
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t = fmaxf(t, red[w]);
    res[qi] = t;
  }
}

// W(q) = v^1/2 eps^-1 v^1/2 (head at q = 0: mini-zone average, wings zero); zero padding to ng_max.
__global__ void w_kernel(DevSys d, const float2* __restrict__ X, float2* __restrict__ W, int q_begin, float head) {
  const int qi = blockIdx.y, q = q_begin + qi;
  const int NG = d.ngq[q];
  const float2* Xq = X + (size_t)qi * d.ng_max * d.ng_max;
  float2* Wq = W + (size_t)q * d.ng_max * d.ng_max;
  const float* vs = d.vsq + (size_t)q * d.ng_max;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < (long long)d.ng_max * d.ng_max;
       i += (long long)gridDim.x * blockDim.x) {
    const int r = (int)(i / d.ng_max), c = (int)(i % d.ng_max);
    float2 v = make_float2(0.f, 0.f);
    if (r < NG && c < NG) {
      const float2 x = Xq[i];
      if (q == 0 && (r == 0 || c == 0)) {
        if (r == 0 && c == 0) v = make_float2(x.x * head, x.y * head);
      } else {
        const float f = vs[r] * vs[c];
        v = make_float2(x.x * f, x.y * f);
      }
    }
    Wq[i] = v;
  }
}

}  // namespace

namespace {
size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

struct ScreenWs {                                 // eps, X, T; images of eps, X (128-row tiles), T; of the pair vectors of q_images q
  size_t E, X, T, img[3], inv[3], vimg, vinv, sw, R, total;
};
ScreenWs layout(const DevSys& d, long long nq) {
  const size_t mat = a256((size_t)nq * d.ng_max * d.ng_max * sizeof(float2)), vec = a256((size_t)nq * d.ng_max * 4);
  const int K = d.nkpt * d.nv * d.nc;
  ScreenWs w;
  size_t o = 0;
  w.E = o; o += mat;
  w.X = o; o += mat;
  w.T = o; o += mat;
  for (int i = 0; i < 3; ++i) {
    w.img[i] = o; o += a256(nq * qgeo(d, d.ng_max, i == 1 ? kTM : tcf::n_tile(d.ng_max)).batch);
    w.inv[i] = o; o += vec;
  }
  w.vimg = o; o += a256((size_t)std::min<long long>(nq, q_images(d)) * qgeo(d, K, kTM).batch);
  w.vinv = o; o += vec;
  w.sw = o; o += a256((size_t)nq * K * 4);
  w.R = o; o += a256((size_t)nq * 4);
  w.total = o;
  return w;
}
}  // namespace

size_t screen_ws_bytes(const DevSys& d, long long qchunk) { return kWsSlack + layout(d, qchunk).total; }

int launch_screening(const DevSys& d, void* rho_chi, const double* energies, const void* P, int q_begin, int q_end,
                     int iterations, void* W, float* residual, void* ws, double gap_floor, int* status, void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  const int nq = q_end - q_begin, K = d.nkpt * d.nv * d.nc;
  const long long rows = (long long)nq * K;
  const ScreenWs L = layout(d, nq);
  unsigned char* base = ws_base(ws);
  float2* E = (float2*)(base + L.E);
  float2* X = (float2*)(base + L.X);
  float2* T = (float2*)(base + L.T);
  unsigned char* img[3];
  float* inv[3];
  for (int i = 0; i < 3; ++i) {
    img[i] = (unsigned char*)(base + L.img[i]);
    inv[i] = (float*)(base + L.inv[i]);
  }
  unsigned char* vimg = (unsigned char*)(base + L.vimg);
  float* vinv = (float*)(base + L.vinv);
  float* sw = (float*)(base + L.sw);
  unsigned* R = (unsigned*)(base + L.R);
  float2* a = (float2*)rho_chi;
  // scaled pair vectors and the largest component of each of their columns
  int e = (int)cudaMemsetAsync(vinv, 0, (size_t)nq * d.ng_max * 4, st);
  if (!e) e = (int)cudaMemsetAsync(R, 0, (size_t)nq * 4, st);
  if (e) return e;
  weight_kernel<<<(unsigned)((rows + 255) / 256), 256, 0, st>>>(d, energies, q_begin, rows, gap_floor, sw);
  scale_kernel<<<dim3((K + kScaleRows - 1) / kScaleRows, nq), 256, 0, st>>>(d, a, sw, (const double2*)P, q_begin, K,
                                                                          (unsigned*)vinv);
  const long long nv = (long long)nq * d.ng_max;
  tcf::inv_scale_kernel<<<(unsigned)((nv + 255) / 256), 256, 0, st>>>((unsigned*)vinv, nv);
  // eps = I + A^T conj(A), q_images q at a time
  const QGeo gv = qgeo(d, K, kTM), g = qgeo(d, d.ng_max, kTM), gb = qgeo(d, d.ng_max, tcf::n_tile(d.ng_max));
  const int qi = q_images(d);
  for (int q0 = 0; q0 < nq; q0 += qi) {
    const int nb = std::min(qi, nq - q0);
    const float2* aq = a + (size_t)q0 * K * d.ng_max;
    const float* iq = vinv + (size_t)q0 * d.ng_max;
    tcf::split_cols_kernel<<<dim3((d.ng_max + tcf::kColG - 1) / tcf::kColG, gv.kc, nb), tcf::kColThreads, 0, st>>>(
        VecSrc{d.ngq, aq, q_begin + q0, K, d.ng_max, nb}, iq, vimg, gv.batch, kTM, gv.kc);
    if ((e = (int)cudaGetLastError())) return e;
    QOp<0> op{d.ngq, gv, gv, vimg, vimg, iq, iq, E + (size_t)q0 * d.ng_max * d.ng_max, q_begin + q0, K, 0.f, 0.f, status,
              (long long)nb * gv.nt * gv.nt};
    if ((e = tcf::launch(op, stream))) return e;
  }
  gershgorin_kernel<<<dim3((d.ng_max + 7) / 8, nq), 256, 0, st>>>(d, E, R, q_begin);
  ns_init_kernel<<<dim3(32, nq), 256, 0, st>>>(d, R, X, q_begin);
  const long long nt = (long long)nq * g.nt * gb.nt;
  if ((e = split_matrix(d, gb, E, img[0], inv[0], q_begin, nq, st))) return e;
  for (int it = 0; it < iterations; ++it) {
    if ((e = split_matrix(d, g, X, img[1], inv[1], q_begin, nq, st))) return e;
    QOp<1> t{d.ngq, g, gb, img[1], img[0], inv[1], inv[0], T, q_begin, 0, 2.f, -1.f, status, nt};      // T = 2 I - X eps
    if ((e = tcf::launch(t, stream))) return e;
    if ((e = split_matrix(d, gb, T, img[2], inv[2], q_begin, nq, st))) return e;
    QOp<2> y{d.ngq, g, gb, img[1], img[2], inv[1], inv[2], X, q_begin, 0, 0.f, 1.f, status, nt};       // X <- X T^H
    if ((e = tcf::launch(y, stream))) return e;
  }
  if (residual) {
    if ((e = split_matrix(d, g, X, img[1], inv[1], q_begin, nq, st))) return e;
    QOp<1> t{d.ngq, g, gb, img[1], img[0], inv[1], inv[0], T, q_begin, 0, 0.f, 1.f, status, nt};       // T = X eps = (eps X)^H
    if ((e = tcf::launch(t, stream))) return e;
    residual_kernel<<<nq, 256, 0, st>>>(d, T, residual, q_begin);
  }
  const double qc = cbrt(6.0 * kPi * kPi / (d.omega_cell * d.nkpt));
  const float head = (float)(12.0 * kPi / (qc * qc));
  w_kernel<<<dim3(64, nq), 256, 0, st>>>(d, X, (float2*)W, q_begin, head);
  return (int)cudaGetLastError();
}

}  // namespace bse
