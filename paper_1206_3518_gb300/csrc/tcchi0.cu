// The optical-limit response chi~0(w) of TDDFT (tddft.cu has the Dyson equation and the ALDA kernel):
//
//   chi~0_GG'(w) = 2/(Omega Nk) sum_S [ r_S(w) a_S(G) conj a_S(G') + rb_S(w) abar_S(G) conj abar_S(G') ],
//   r = 1/(w - de + i eta),  rb = -1/(w + de + i eta),  a_S(G) = v^1/2(G) rho_vc^{kk}(G),  a_S(0) = sqrt(4 pi) conj(P_S),
//   abar_S(G) = conj(a_S(-G)),  abar_S(0) = -conj(a_S(0)).
//
// Only the weights depend on w, and T_S(G, G') = a_S(G) conj a_S(G') is Hermitian, so for all frequencies
// together the sums are one real product
//
//   Z[(w, j)][(G <= G', t)] = sum_S R_j(w, S) T_t(S, G, G'),   R_j = Re r, Im r, Re rb, Im rb;  T_t = Re T, Im T:
//
// half the multiply-adds of a complex product per frequency and per term (the second term is T at (-G', -G)), as
// FP16x3 with promoted accumulation (tcf16.cuh, real products).  T is formed in FP32 and split into images a panel of
// pairs at a time, the weights (FP64) 1024 frequencies at a time; Z of 128 frequencies is combined into
// chi~0 by two passes, one per term (each touches every element of chi~0 at most once).
//
// Measured, fcc 8x8x8 3v4c (307 G, 6144 transitions), 1000 frequencies: 14.7 ms (products 10.2, combination
// 3.3, images 0.9), error against 64 bits (2-norm) 2.4e-7; a weighted complex Gram product per frequency on the FP32
// pipes took 327.6 ms, 1.2e-6.
#include <cuda_runtime.h>

#include <algorithm>

#include "internal.h"
#include "tcf16.cuh"

namespace bse {
namespace {

constexpr int kW = 1024, kWZ = 128;              // frequencies per weights image, per Z
constexpr int kWPer = 4;                         // frequencies per thread of combine_kernel
constexpr size_t kPanelBytes = size_t(1) << 29;  // images of T and rows of Z at a time
constexpr long long kWave = 38 * 128;            // pairs of one tile for every SM (4 kWZ / 128 row tiles each)
constexpr size_t kRowB = umma::kRow;

size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

struct Geo {
  int ng, dim, kc, sp;                           // S chunks of 64, padded length
  long long pairs, panel;                        // G <= G' pairs, pairs per panel (a multiple of 128)
  size_t o_a, o_amax, o_de, o_w, o_invw, o_t, o_invt, o_z, total;
};

Geo geo_of(const DevSys& d) {
  Geo g;
  g.ng = d.ng0;
  g.dim = d.dim;
  g.kc = (d.dim + tcf::kRealK - 1) / tcf::kRealK;
  g.sp = g.kc * tcf::kRealK;
  g.pairs = (long long)g.ng * (g.ng + 1) / 2;
  const size_t per_pair = (size_t)g.kc * 4 * kRowB;           // two rows, hi and lo
  const size_t per_z = (size_t)4 * kWZ * 2 * sizeof(float);   // a pair's columns of Z
  g.panel = std::max<long long>(1, (long long)(kPanelBytes / ((per_pair + per_z) * 128))) * 128;
  if (g.panel > kWave) g.panel -= g.panel % kWave;            // whole waves of tiles
  g.panel = std::min(g.panel, (g.pairs + 127) / 128 * 128);
  size_t o = 0;
  g.o_a = o; o = a256(o + (size_t)g.ng * g.sp * sizeof(float2));
  g.o_amax = o; o = a256(o + (size_t)g.ng * sizeof(float));
  g.o_de = o; o = a256(o + (size_t)g.dim * sizeof(double));
  g.o_w = o; o = a256(o + (size_t)(4 * kW / tcf::kTM) * g.kc * 2 * tcf::kTileA);
  g.o_invw = o; o = a256(o + (size_t)4 * kW * sizeof(float));
  g.o_t = o; o = a256(o + (size_t)g.panel * per_pair);
  g.o_invt = o; o = a256(o + (size_t)2 * g.panel * sizeof(float));
  g.o_z = o; o = a256(o + (size_t)4 * kWZ * 2 * g.panel * sizeof(float));
  g.total = o;
  return g;
}

// a [ng][sp] (transposed, zero past dim), its largest component per G, and de [dim].  One CTA per G.
__global__ __launch_bounds__(256) void pair_vectors_kernel(DevSys d, const float2* __restrict__ rho_x,
                                                           const double2* __restrict__ P, const double* __restrict__ e,
                                                           double delta, int sp, float2* __restrict__ a,
                                                           float* __restrict__ amax, double* __restrict__ de) {
  const int G = blockIdx.x;
  const float s4pi = 3.5449077018110318f;        // sqrt(4 pi)
  const float vs = d.vsq[G];                     // q = 0 row: sqrt(4 pi)/|G|
  float m = 0.f;
  for (int S = threadIdx.x; S < sp; S += blockDim.x) {
    float2 x = make_float2(0.f, 0.f);
    if (S < d.dim) {
      if (G == 0) {
        const double2 p = P[S];
        x = make_float2(s4pi * (float)p.x, -s4pi * (float)p.y);
        const int nvc = d.nv * d.nc, k = S / nvc, v = (S / d.nc) % d.nv, c = S % d.nc;
        de[S] = e[(size_t)k * d.nb + d.nv + c] + delta - e[(size_t)k * d.nb + v];
      } else {
        const float2 r = rho_x[(size_t)S * d.ng_max + G];
        x = make_float2(vs * r.x, vs * r.y);
      }
    }
    a[(size_t)G * sp + S] = x;
    m = fmaxf(m, fmaxf(fabsf(x.x), fabsf(x.y)));
  }
  __shared__ float red[8];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < 8; ++i) m = fmaxf(m, red[i]);
    amax[G] = m;
  }
}

__device__ __forceinline__ long long row_pairs(int G, int ng) { return (long long)G * ng - (long long)G * (G - 1) / 2; }
// pair p -> (G, G' >= G), row by row
__device__ __forceinline__ void pair_of(long long p, int ng, int& G, int& G2) {
  const float b = 2.f * ng + 1.f;                // an estimate: the loops correct it
  int g = (int)(0.5f * (b - sqrtf(fmaxf(b * b - 8.f * (float)p, 0.f))));
  g = g < 0 ? 0 : (g > ng - 1 ? ng - 1 : g);
  while (g > 0 && row_pairs(g, ng) > p) --g;
  while (g + 1 < ng && row_pairs(g + 1, ng) <= p) ++g;
  G = g;
  G2 = g + (int)(p - row_pairs(g, ng));
}

__device__ __forceinline__ void put8_real(unsigned char* hi, unsigned char* lo, int r, int oct, const float (&x)[8]) {
  uint4 h, l;
  tcf::split_pair(x[0], x[1], h.x, l.x);
  tcf::split_pair(x[2], x[3], h.y, l.y);
  tcf::split_pair(x[4], x[5], h.z, l.z);
  tcf::split_pair(x[6], x[7], h.w, l.w);
  *reinterpret_cast<uint4*>(hi + umma::swz(r, oct)) = h;
  *reinterpret_cast<uint4*>(lo + umma::swz(r, oct)) = l;
}

// Images of T for pairs p0 .. p0 + np: rows 2 i (Re) and 2 i + 1 (Im) of tiles of 256 rows.  Eight lanes per pair and
// chunk, chunks blockIdx.y, + gridDim.y, ...  The scale comes from max |a(G)| max |a(G')|, a bound of max_S |T| (a few
// powers of two above it, which FP16 has to spare).
__global__ __launch_bounds__(256) void t_images_kernel(int ng, int sp, int kc, const float2* __restrict__ a,
                                                       const float* __restrict__ amax, long long p0, long long np,
                                                       unsigned char* __restrict__ img, float* __restrict__ inv) {
  const long long i = (long long)blockIdx.x * 32 + (threadIdx.x >> 3);
  const int oct = threadIdx.x & 7;
  if (i >= np) return;
  int G, G2;
  pair_of(p0 + i, ng, G, G2);
  const int e = tcf::scale_exp(2.f * amax[G] * amax[G2]);
  const float sc = tcf::pow2(e);
  if (blockIdx.y == 0 && oct < 2) inv[2 * i + oct] = tcf::pow2(-e);
  constexpr size_t lo = tcf::kRealN * kRowB;
  const int r = (int)((2 * i) % tcf::kRealN);
  unsigned char* tile = img + (size_t)((2 * i) / tcf::kRealN) * kc * (2 * lo);
  for (int c = blockIdx.y; c < kc; c += gridDim.y) {
    const float4* x = reinterpret_cast<const float4*>(a + (size_t)G * sp + c * tcf::kRealK + 8 * oct);
    const float4* y = reinterpret_cast<const float4*>(a + (size_t)G2 * sp + c * tcf::kRealK + 8 * oct);
    float tr[8], ti[8];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float4 p = x[u], q = y[u];
      tr[2 * u] = (p.x * q.x + p.y * q.y) * sc;               // a conj(a')
      ti[2 * u] = (p.y * q.x - p.x * q.y) * sc;
      tr[2 * u + 1] = (p.z * q.z + p.w * q.w) * sc;
      ti[2 * u + 1] = (p.w * q.z - p.z * q.w) * sc;
    }
    unsigned char* hi = tile + (size_t)c * (2 * lo);
    put8_real(hi, hi + lo, r, oct, tr);
    put8_real(hi, hi + lo, r + 1, oct, ti);
  }
}

// Images of the weights of nw frequencies: rows 4 w + j.  One CTA per frequency.
__global__ __launch_bounds__(256) void weights_kernel(int dim, int kc, const double* __restrict__ de,
                                                      const double* __restrict__ omega, double eta,
                                                      unsigned char* __restrict__ img, float* __restrict__ inv) {
  const int w = blockIdx.x;
  const double om = omega[w];
  // largest |weight| of each row, in FP32 (it only sets a power of two)
  float m[4] = {0.f, 0.f, 0.f, 0.f};
  const float ef = (float)eta;
  for (int S = threadIdx.x; S < dim; S += blockDim.x) {
    const float u = (float)(om - de[S]), v = (float)(om + de[S]);
    const float iu = 1.f / (u * u + ef * ef), iv = 1.f / (v * v + ef * ef);
    m[0] = fmaxf(m[0], fabsf(u) * iu);
    m[1] = fmaxf(m[1], ef * iu);
    m[2] = fmaxf(m[2], fabsf(v) * iv);
    m[3] = fmaxf(m[3], ef * iv);
  }
  __shared__ float red[8][4];
  __shared__ float sc[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m[j] = fmaxf(m[j], __shfl_xor_sync(0xffffffffu, m[j], o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][j] = m[j];
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    float t = 0.f;
    for (int i = 0; i < 8; ++i) t = fmaxf(t, red[i][threadIdx.x]);
    // one power of two less than the largest allows: the FP32 estimate may round down across a power of two
    const int e = tcf::scale_exp(2.f * t);
    sc[threadIdx.x] = tcf::pow2(e);
    inv[4 * w + threadIdx.x] = tcf::pow2(-e);
  }
  __syncthreads();
  const int row = 4 * w;
  unsigned char* tile = img + (size_t)(row / tcf::kTM) * kc * (2 * tcf::kTileA);
  for (int t = threadIdx.x; t < 8 * kc; t += blockDim.x) {
    const int c = t >> 3, oct = t & 7;
    float x[4][8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int S = c * tcf::kRealK + 8 * oct + i;
      double r0 = 0.0, r1 = 0.0, r2 = 0.0, r3 = 0.0;
      if (S < dim) {
        const double u = om - de[S], v = om + de[S];
        const double iu = 1.0 / (u * u + eta * eta), iv = 1.0 / (v * v + eta * eta);
        r0 = u * iu;                              // 1/(w - de + i eta)
        r1 = -eta * iu;
        r2 = -v * iv;                             // -1/(w + de + i eta)
        r3 = eta * iv;
      }
      x[0][i] = (float)r0 * sc[0];
      x[1][i] = (float)r1 * sc[1];
      x[2][i] = (float)r2 * sc[2];
      x[3][i] = (float)r3 * sc[3];
    }
    unsigned char* hi = tile + (size_t)c * (2 * tcf::kTileA);
#pragma unroll
    for (int j = 0; j < 4; ++j) put8_real(hi, hi + tcf::kTileA, row % tcf::kTM + j, oct, x[j]);
  }
}

struct ZOp {
  static constexpr bool kReal = true, kConj = false, kHerm = false;
  const unsigned char *a, *b;
  const float *inva, *invb;
  float* Z;
  int M, K, kc, mt;
  long long N, ldz;
  int* status;
  long long ntiles;
  // row tiles fastest: the CTAs in flight share a panel tile of T, which is read once from memory
  __device__ __forceinline__ bool tile(long long ti, tcf::Tile& o) const {
    const long long nt = ti / mt;
    const int m = (int)(ti - nt * mt);
    o.a_step = 2 * tcf::kTileA;
    o.b_step = (uint32_t)(2 * tcf::kRealN * kRowB);
    o.a = a + (size_t)m * kc * o.a_step;
    o.b = b + (size_t)nt * kc * o.b_step;
    o.K = K;
    o.n = tcf::kRealN;
    o.m0 = m * tcf::kTM;
    o.n0 = 0;
    o.row0 = nt * tcf::kRealN;                    // first column
    o.mvalid = M - o.m0;
    o.nvalid = (int)(N - o.row0 < tcf::kRealN ? N - o.row0 : tcf::kRealN);
    o.batch = 0;
    return true;
  }
  __device__ __forceinline__ float* row_out(const tcf::Tile& t, int row) const {
    return Z + (size_t)(t.m0 + row) * ldz + t.row0;
  }
  __device__ __forceinline__ float row_scale(const tcf::Tile& t, int row) const { return inva[t.m0 + row]; }
  __device__ __forceinline__ float col_scale(const tcf::Tile& t, int col) const { return invb[t.row0 + col]; }
};

// chi[w] +-= the resonant (ANTI = false) or anti-resonant term of pairs p0 .. p0 + np from Z; FIRST: assigned, not added
// (the resonant pass of a panel that holds every pair).
template <bool ANTI, bool FIRST>
__global__ __launch_bounds__(256) void combine_kernel(int ng, const int* __restrict__ gm, long long p0, long long np,
                                                      const float* __restrict__ Z, long long ldz, float pref,
                                                      int nz, float2* __restrict__ chi) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= np) return;
  int G, G2;
  pair_of(p0 + i, ng, G, G2);
  int r1 = G, c1 = G2, r2 = G2, c2 = G;          // r T goes to (r1, c1), r conj(T) to (r2, c2)
  if (ANTI) {                                    // abar(X) conj abar(Y) = +- T(-Y, -X), minus where one of X, Y is 0
    const int m1 = gm[G], m2 = gm[G2];
    r1 = m2;
    c1 = m1;
    r2 = m1;
    c2 = m2;
    if ((m1 == 0) != (m2 == 0)) pref = -pref;
  }
  for (int w = blockIdx.y * kWPer; w < min(nz, (int)(blockIdx.y + 1) * kWPer); ++w) {
    const float2 zr = *reinterpret_cast<const float2*>(Z + (size_t)(4 * w + (ANTI ? 2 : 0)) * ldz + 2 * i);
    const float2 zi = *reinterpret_cast<const float2*>(Z + (size_t)(4 * w + (ANTI ? 3 : 1)) * ldz + 2 * i);
    const float2 x = make_float2(zr.x - zi.y, zr.y + zi.x), y = make_float2(zr.x + zi.y, zi.x - zr.y);
    float2* c = chi + (size_t)w * ng * ng;
    float2* q = c + (size_t)r1 * ng + c1;
    float2 o = FIRST ? make_float2(0.f, 0.f) : *q;
    *q = make_float2(o.x + pref * x.x, o.y + pref * x.y);
    if (G != G2) {
      q = c + (size_t)r2 * ng + c2;
      o = FIRST ? make_float2(0.f, 0.f) : *q;
      *q = make_float2(o.x + pref * y.x, o.y + pref * y.y);
    }
  }
}

}  // namespace

size_t chi0_ws_bytes(const DevSys& d) { return kWsSlack + geo_of(d).total; }

int launch_chi0_optical(const DevSys& d, const void* rho_x, const void* P, const double* energies, double delta,
                        const double* omega, int nw, double eta, void* chi0, void* ws, int* status, void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  const Geo g = geo_of(d);
  unsigned char* base = ws_base(ws);
  float2* a = (float2*)(base + g.o_a);
  float* amax = (float*)(base + g.o_amax);
  double* de = (double*)(base + g.o_de);
  unsigned char* wimg = (unsigned char*)(base + g.o_w);
  float* invw = (float*)(base + g.o_invw);
  unsigned char* timg = (unsigned char*)(base + g.o_t);
  float* invt = (float*)(base + g.o_invt);
  float* Z = (float*)(base + g.o_z);
  float2* chi = (float2*)chi0;
  if (nw <= 0) return 0;
  pair_vectors_kernel<<<g.ng, 256, 0, st>>>(d, (const float2*)rho_x, (const double2*)P, energies, delta, g.sp, a, amax, de);
  int e = (int)cudaGetLastError();
  if (e) return e;
  const bool one = g.panel >= g.pairs;
  if (!one && (e = (int)cudaMemsetAsync(chi, 0, (size_t)nw * g.ng * g.ng * sizeof(float2), st))) return e;
  const float pref = (float)(2.0 * d.norm);
  for (long long p0 = 0; p0 < g.pairs; p0 += g.panel) {
    const long long np = std::min(g.panel, g.pairs - p0);
    const unsigned bx = (unsigned)((np + 31) / 32), by = bx >= 2048 ? 1u : (unsigned)std::min<long long>(g.kc, 2048 / bx + 1);
    t_images_kernel<<<dim3(bx, by), 256, 0, st>>>(g.ng, g.sp, g.kc, a, amax, p0, np, timg, invt);
    if ((e = (int)cudaGetLastError())) return e;
    for (int w0 = 0; w0 < nw; w0 += kW) {
      const int nwi = std::min(kW, nw - w0);
      if (p0 == 0 || nw > kW) {                   // one image holds every frequency: made for the first panel only
        weights_kernel<<<nwi, 256, 0, st>>>(g.dim, g.kc, de, omega + w0, eta, wimg, invw);
        if ((e = (int)cudaGetLastError())) return e;
      }
      for (int z0 = 0; z0 < nwi; z0 += kWZ) {
        const int nz = std::min(kWZ, nwi - z0);
        ZOp op;
        op.a = wimg + (size_t)(4 * z0 / tcf::kTM) * g.kc * 2 * tcf::kTileA;
        op.b = timg;
        op.inva = invw + 4 * z0;
        op.invb = invt;
        op.Z = Z;
        op.M = 4 * nz;
        op.N = 2 * np;
        op.K = g.dim;
        op.kc = g.kc;
        op.mt = (op.M + tcf::kTM - 1) / tcf::kTM;
        op.ldz = 2 * g.panel;
        op.status = status;
        op.ntiles = (long long)op.mt * ((op.N + tcf::kRealN - 1) / tcf::kRealN);
        if ((e = tcf::launch(op, stream))) return e;
        float2* c = chi + (size_t)(w0 + z0) * g.ng * g.ng;
        const dim3 grid((unsigned)((np + 255) / 256), (nz + kWPer - 1) / kWPer);
        if (one)
          combine_kernel<false, true><<<grid, 256, 0, st>>>(g.ng, d.gminus0, p0, np, Z, op.ldz, pref, nz, c);
        else
          combine_kernel<false, false><<<grid, 256, 0, st>>>(g.ng, d.gminus0, p0, np, Z, op.ldz, pref, nz, c);
        combine_kernel<true, false><<<grid, 256, 0, st>>>(g.ng, d.gminus0, p0, np, Z, op.ldz, pref, nz, c);
        if ((e = (int)cudaGetLastError())) return e;
      }
    }
  }
  return 0;
}

}  // namespace bse
