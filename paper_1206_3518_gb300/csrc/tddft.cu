// Macroscopic dielectric function from TDDFT with local fields (Sec. II A-B: Eqs. chi0_GG, Dyson_GG,
// epsilon_-1, epsilon_M) in the optical limit q -> 0, on the q = 0 sphere of the system.
//
//   chi~0_GG'(w) = 2/(Omega Nk) sum_S [ a_S(G) conj a_S(G') / (w - de_S + i eta)
//                                      - abar_S(G) conj abar_S(G') / (w + de_S + i eta) ]
//   a_S(G) = v^1/2(G) rho_vc^{kk}(G),  abar_S(G) = v^1/2(G) conj(rho_vc^{kk}(-G))   (G != 0)
//   a_S(0) = sqrt(4 pi) conj(P_S),     abar_S(0) = -sqrt(4 pi) P_S                   (k.p limit)
//   eps^-1 = I + (I - chi~0 (I + F))^-1 chi~0,   eps_M = 1/[eps^-1]_00
//
// F = v^-1/2 f_xc v^-1/2 is zero for the RPA and the adiabatic local-density kernel otherwise:
// f_xc(r) = d^2(n eps_xc)/dn^2 at the density n(r) = 2/(Omega Nk) sum_{k,v} |u_vk(r)|^2 (Slater
// exchange + Perdew-Zunger correlation), F_GG' = |G| f_xc(G - G') |G'|/(4 pi).
//
// Kernels here (chi~0(w) is in tcchi0.cu): the density, f_xc(r) and its transform onto the difference box of the sphere
// (three separable direct DFT passes in FP64); the batched Dyson solve: M = I - chi~0 (I + F) augmented with
// chi~0 e_0, Gaussian elimination with partial pivoting and back substitution, one CTA per frequency (FP32 matrix,
// FP64 result).  No device-side waits; capturable.
#include <cuda_runtime.h>

#include <cstdint>

#include "internal.h"

namespace bse {
namespace {

// Complex products of the Dyson solve with their roundings spelled out (left to the compiler's contraction they change
// with the code around them, and eps_M is returned in FP64).
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -__fmul_rn(a.y, b.y)), fmaf(a.y, b.x, __fmul_rn(a.x, b.y)));
}
__device__ __forceinline__ float2 cmul_f(float2 a, float2 b) {   // of the product with the kernel F
  return make_float2(fmaf(a.x, b.x, -__fmul_rn(a.y, b.y)), fmaf(a.x, b.y, __fmul_rn(a.y, b.x)));
}

// [M | b] rows of every frequency with a kernel F: M = I - (chi~0 + chi~0 F), b = chi~0 e_0 (row stride n + 1).  The rows
// of all frequencies are one product with F: 128 x 64 tiles, 8 x 4 outputs a thread, k in ascending order.
// Bound by the FP32 pipes (a complex multiply-add is six instructions in the order that the result has always been
// rounded in; 307 x 307, 2000 frequencies 13.1 ms; per frequency,
// with 4 x 4 outputs a thread and a product array, 13.8 + 0.8 ms).
namespace gf {
constexpr int TM = 128, TN = 64, TK = 16, kThreads = 256;
}
__global__ void __launch_bounds__(gf::kThreads, 2) kernel_rows_kernel(int n, long long rows, const float2* __restrict__ chi,
                                                                     const float2* __restrict__ F,
                                                                     float2* __restrict__ aug) {
  using namespace gf;
  __shared__ __align__(16) float2 sa[2][TK][TM], sb[2][TK][TN];
  const long long r0 = (long long)blockIdx.y * TM;
  const int c0 = blockIdx.x * TN, t = threadIdx.x, tm = t >> 4, tn = t & 15;
  // staging: A row t / 2, eight k; B k t / 16, four columns
  const int ar = t >> 1, ak = (t & 1) * 8, bk = t >> 4, bc = (t & 15) * 4;
  const float2* Ap = chi + (size_t)(r0 + ar) * n;
  const bool a_in = r0 + ar < rows;
  float2 ra[8], rb[4];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int i = 0; i < 8; ++i) ra[i] = (a_in && k0 + ak + i < n) ? Ap[k0 + ak + i] : make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < 4; ++i)
      rb[i] = (k0 + bk < n && c0 + bc + i < n) ? F[(size_t)(k0 + bk) * n + c0 + bc + i] : make_float2(0.f, 0.f);
  };
  auto put = [&](int buf) {
#pragma unroll
    for (int i = 0; i < 8; ++i) sa[buf][ak + i][ar] = ra[i];
#pragma unroll
    for (int i = 0; i < 4; ++i) sb[buf][bk][bc + i] = rb[i];
  };
  float2 acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
  fetch(0);
  put(0);
  __syncthreads();
  int buf = 0;
  for (int k0 = 0; k0 < n; k0 += TK) {
    const bool more = k0 + TK < n;
    if (more) fetch(k0 + TK);
#pragma unroll 4
    for (int k = 0; k < TK; ++k) {
      float2 x[8], y[4];
      const float4* px = reinterpret_cast<const float4*>(&sa[buf][k][tm * 8]);
      const float4* py = reinterpret_cast<const float4*>(&sb[buf][k][tn * 4]);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float4 v = px[i];
        x[2 * i] = make_float2(v.x, v.y);
        x[2 * i + 1] = make_float2(v.z, v.w);
      }
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const float4 v = py[i];
        y[2 * i] = make_float2(v.x, v.y);
        y[2 * i + 1] = make_float2(v.z, v.w);
      }
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float2 p = cmul_f(x[i], y[j]);
          acc[i][j].x = __fadd_rn(acc[i][j].x, p.x);
          acc[i][j].y = __fadd_rn(acc[i][j].y, p.y);
        }
    }
    if (more) {
      put(buf ^ 1);
      __syncthreads();
      buf ^= 1;
    }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const long long r = r0 + tm * 8 + i;
    if (r >= rows) continue;
    const int ri = (int)(r % n);
    const float2* cr = chi + (size_t)r * n;
    float2* out = aug + (size_t)r * (n + 1);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int c = c0 + tn * 4 + j;
      if (c >= n) continue;
      float2 v = cr[c];
      v.x += acc[i][j].x;
      v.y += acc[i][j].y;
      out[c] = make_float2((ri == c ? 1.f : 0.f) - v.x, -v.y);
    }
    if (c0 == 0 && tn == 0) out[n] = cr[0];
  }
}

// The same without a kernel: M = I - chi~0.
__global__ void augment_kernel(int n, int nw, const float2* __restrict__ chi, float2* __restrict__ aug) {
  const long long total = (long long)nw * n * (n + 1);
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total; t += (long long)gridDim.x * blockDim.x) {
    const int w = (int)(t / ((long long)n * (n + 1)));
    const long long rem = t - (long long)w * n * (n + 1);
    const int i = (int)(rem / (n + 1)), j = (int)(rem - (long long)i * (n + 1));
    const float2* cw = chi + (size_t)w * n * n;
    float2 v;
    if (j == n) {
      v = cw[(size_t)i * n];
    } else {
      const float2 c = cw[(size_t)i * n + j];
      v = make_float2((i == j ? 1.f : 0.f) - c.x, -c.y);
    }
    aug[t] = v;
  }
}

// One CTA per frequency: Gaussian elimination with partial pivoting on [M | b], back substitution for x,
// eps_M = 1/(1 + x_0).
//
// Blocked by panels of PB columns held in shared memory: the rest of the matrix is read and written once per panel
// (n^3/(3 PB) elements of 16 bytes) instead of once per column, its PB updates running in registers.  Every element
// sees the same operations in the same order as in the unblocked elimination (the updates by ascending column, the
// row swaps in their order), so the result is the same bit for bit.  Measured, 307 x 307, 2000 frequencies: column by
// column 62.8 ms, by panels of 16 15.3 ms.
constexpr int kSolveThreads = 512, kSolveVirtual = 1024;   // threads; threads that the back substitution's sums are split over

__device__ __forceinline__ void csub_mul(float2& v, float2 l, float2 u) {
  const float2 p = cmul(l, u);
  v.x = __fsub_rn(v.x, p.x);
  v.y = __fsub_rn(v.y, p.y);
}

template <int PB>
__global__ void __launch_bounds__(kSolveThreads, 2) dyson_solve_kernel(int n, float2* __restrict__ aug,
                                                                   double2* __restrict__ eps_m,
                                                                   float2* __restrict__ xbuf) {
  const int w = blockIdx.x, ld = n + 1, tid = threadIdx.x, nt = kSolveThreads;
  float2* M = aug + (size_t)w * n * ld;
  float2* x = xbuf + (size_t)w * n;
  __shared__ float red_v[32], red_w[32];
  __shared__ int red_i[32];
  __shared__ int piv[PB];
  __shared__ float2 pivrow_inv;
  extern __shared__ float2 dyn[];
  constexpr int LP = PB + 1;
  float2* pan = dyn;                              // [n - kb][LP]: the panel, multipliers below its diagonal
  float2* U = dyn + (size_t)n * LP;               // [PB][ld]: the panel's rows right of it
  for (int kb = 0; kb < n; kb += PB) {
    const int pw = min(PB, n - kb), nr = n - kb;
    for (int t = tid; t < nr * PB; t += nt) {
      const int r = t / PB, c = t - r * PB;
      if (c < pw) pan[r * LP + c] = M[(size_t)(kb + r) * ld + kb + c];
    }
    __syncthreads();
    for (int kk = 0; kk < pw; ++kk) {
      // pivot: largest |M[i][k]|, i >= k (the lowest row of equal ones)
      float best = -1.f;
      int bi = kk;
      for (int i = kk + tid; i < nr; i += nt) {
        const float2 v = pan[i * LP + kk];
        const float m = v.x * v.x + v.y * v.y;
        if (m > best) { best = m; bi = i; }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
      }
      if ((tid & 31) == 0) { red_v[tid >> 5] = best; red_i[tid >> 5] = bi; }
      __syncthreads();
      if (tid < 32) {
        best = tid < (nt >> 5) ? red_v[tid] : -1.f;
        bi = tid < (nt >> 5) ? red_i[tid] : kk;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const float ob = __shfl_xor_sync(0xffffffffu, best, o);
          const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
          if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
        }
        if (tid == 0) piv[kk] = bi;
        if (bi != kk && tid < pw) {               // swap the panel's rows (every lane has the winner)
          const float2 t0 = pan[kk * LP + tid];
          pan[kk * LP + tid] = pan[bi * LP + tid];
          pan[bi * LP + tid] = t0;
        }
        __syncwarp();
        if (tid == 0) {
          const float2 d = pan[kk * LP + kk];
          const float m = d.x * d.x + d.y * d.y;
          pivrow_inv = make_float2(d.x / m, -d.y / m);
        }
      }
      __syncthreads();
      const float2 inv = pivrow_inv;
      for (int i = kk + 1 + tid; i < nr; i += nt) {
        const float2 l = cmul(pan[i * LP + kk], inv);
        pan[i * LP + kk] = l;
        for (int c = kk + 1; c < pw; ++c) {
          float2 v = pan[i * LP + c];
          csub_mul(v, l, pan[kk * LP + c]);
          pan[i * LP + c] = v;
        }
      }
      __syncthreads();
    }
    // the panel's own rows of U, and right of the panel: swaps, then the rows of U (one thread per column)
    for (int t = tid; t < pw * pw; t += nt) {
      const int r = t / pw, c = t - r * pw;
      if (c >= r) M[(size_t)(kb + r) * ld + kb + c] = pan[r * LP + c];
    }
    const int j0 = kb + pw;
    for (int j = j0 + tid; j <= n; j += nt) {
      for (int kk = 0; kk < pw; ++kk) {
        const int p = piv[kk];
        if (p != kk) {
          const float2 t0 = M[(size_t)(kb + kk) * ld + j];
          M[(size_t)(kb + kk) * ld + j] = M[(size_t)(kb + p) * ld + j];
          M[(size_t)(kb + p) * ld + j] = t0;
        }
      }
      float2 u[PB];
#pragma unroll
      for (int kk = 0; kk < PB; ++kk) {
        if (kk < pw) {
          float2 v = M[(size_t)(kb + kk) * ld + j];
#pragma unroll
          for (int q = 0; q < kk; ++q) csub_mul(v, pan[kk * LP + q], u[q]);
          u[kk] = v;
          M[(size_t)(kb + kk) * ld + j] = v;
          U[kk * ld + j] = v;
        }
      }
    }
    __syncthreads();
    // the rest: four rows of one column per thread and pass, neighbouring threads neighbouring columns
    const int cols = n + 1 - j0, nrow4 = (n - j0 + 3) / 4;
    for (int t = tid; t < nrow4 * cols; t += nt) {
      const int g = t / cols, j = j0 + (t - g * cols), i0 = j0 + 4 * g;
      float2 v[4];
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (i0 + q < n) v[q] = M[(size_t)(i0 + q) * ld + j];
#pragma unroll
      for (int kk = 0; kk < PB; ++kk) {
        if (kk >= pw) break;
        const float2 u = U[kk * ld + j];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (i0 + q < n) csub_mul(v[q], pan[(i0 + q - kb) * LP + kk], u);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (i0 + q < n) M[(size_t)(i0 + q) * ld + j] = v[q];
    }
    __syncthreads();
  }
  // back substitution, one row at a time from the bottom (block reduction of the row's dot product over 1024 partial
  // sums, two per thread)
  for (int i = n - 1; i >= 0; --i) {
#pragma unroll
    for (int h = 0; h < kSolveVirtual / kSolveThreads; ++h) {
      const int vt = tid + h * kSolveThreads;
      float sr = 0.f, si = 0.f;
      for (int j = i + 1 + vt; j < n; j += kSolveVirtual) {
        const float2 m = M[(size_t)i * ld + j], xv = x[j];
        sr += m.x * xv.x - m.y * xv.y;
        si += m.x * xv.y + m.y * xv.x;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        sr += __shfl_xor_sync(0xffffffffu, sr, o);
        si += __shfl_xor_sync(0xffffffffu, si, o);
      }
      if ((tid & 31) == 0) { red_v[vt >> 5] = sr; red_w[vt >> 5] = si; }
    }
    __syncthreads();
    if (tid == 0) {
      float tr = 0.f, ti = 0.f;
      for (int u = 0; u < kSolveVirtual >> 5; ++u) { tr += red_v[u]; ti += red_w[u]; }
      const float2 b = M[(size_t)i * ld + n], d = M[(size_t)i * ld + i];
      const float2 num = make_float2(b.x - tr, b.y - ti);
      const float m = d.x * d.x + d.y * d.y;
      x[i] = make_float2((num.x * d.x + num.y * d.y) / m, (num.y * d.x - num.x * d.y) / m);
    }
    __syncthreads();
  }
  if (tid == 0) {
    const double re = 1.0 + (double)x[0].x, im = (double)x[0].y;
    const double m = re * re + im * im;
    eps_m[w] = make_double2(re / m, -im / m);
  }
}

size_t solve_smem(int n, int pb) { return ((size_t)n * (pb + 1) + (size_t)pb * (n + 1)) * sizeof(float2); }

template <int PB>
int launch_solve(int n, int nw, float2* aug, double2* eps_m, float2* xb, cudaStream_t st) {
  const size_t sm = solve_smem(n, PB);
  if (int e = allow_smem((const void*)dyson_solve_kernel<PB>)) return e;
  dyson_solve_kernel<PB><<<nw, kSolveThreads, sm, st>>>(n, aug, eps_m, xb);
  return (int)cudaGetLastError();
}

// ---------------------------------------------------------------------------- ALDA

__device__ __forceinline__ double lda_fxc(double n) {
  const double kPiD = 3.141592653589793;
  const double fx = -(1.0 / 3.0) * cbrt(3.0 / kPiD) * pow(n, -2.0 / 3.0);
  const double rs = cbrt(3.0 / (4.0 * kPiD * n));
  double d1, d2;
  if (rs >= 1.0) {                               // Perdew-Zunger, gamma / (1 + beta1 sqrt(rs) + beta2 rs)
    const double g = -0.1423, b1 = 1.0529, b2 = 0.3334, sq = sqrt(rs);
    const double D = 1.0 + b1 * sq + b2 * rs, D1 = b1 / (2.0 * sq) + b2, D2 = -b1 / (4.0 * rs * sq);
    d1 = -g * D1 / (D * D);
    d2 = -g * (D2 / (D * D) - 2.0 * D1 * D1 / (D * D * D));
  } else {                                       // A ln rs + B + C rs ln rs + D rs
    const double A = 0.0311, C = 0.0020, Dd = -0.0116;
    d1 = A / rs + C * (log(rs) + 1.0) + Dd;
    d2 = -A / (rs * rs) + C / rs;
  }
  const double fc = -(rs / (3.0 * n)) * ((2.0 / 3.0) * d1 - (rs / 3.0) * d2);
  return fx + fc;
}

// f_xc(r) at every grid point from the valence bands of u(r) in the pair workspace
__global__ void alda_fxc_kernel(DevSys d, const float2* __restrict__ u, double* __restrict__ f, double norm2) {
  const long long nr = (long long)d.n1 * d.n2 * d.n3;
  for (long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x; r < nr; r += (long long)gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int k = 0; k < d.nkpt; ++k)
      for (int v = 0; v < d.nv; ++v) {
        const float2 x = u[((size_t)k * d.nb + v) * nr + r];
        s += (double)x.x * x.x + (double)x.y * x.y;
      }
    const double n = fmax(norm2 * s, 1e-6);
    f[r] = lda_fxc(n);
  }
}

// One separable DFT pass along axis `ax` of a box whose other two extents are (e1, e2):
// out[j][i1][i2] = sum_x in[x][i1][i2] exp(-2 pi i (j - m) x / N), j = 0 .. 2m, in/out indexed with the
// transformed axis first.  Input real (pass 1) or complex.
__global__ void dft_pass_kernel(const double2* __restrict__ in, double2* __restrict__ out, int N, int m, int e1, int e2,
                                int in_stride_ax, int in_stride_1, int in_stride_2, int out_stride_ax,
                                int out_stride_1, int out_stride_2) {
  const long long total = (long long)(2 * m + 1) * e1 * e2;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total; t += (long long)gridDim.x * blockDim.x) {
    const int j = (int)(t / ((long long)e1 * e2));
    const int rem = (int)(t - (long long)j * e1 * e2);
    const int i1 = rem / e2, i2 = rem - i1 * e2;
    const int fq = j - m;
    double sr = 0.0, si = 0.0;
    for (int x = 0; x < N; ++x) {
      const double2 v = in[(size_t)x * in_stride_ax + (size_t)i1 * in_stride_1 + (size_t)i2 * in_stride_2];
      double sn, cs;
      sincospi(-2.0 * (double)(((long long)fq * x) % N) / (double)N, &sn, &cs);
      sr += v.x * cs - v.y * sn;
      si += v.x * sn + v.y * cs;
    }
    out[(size_t)j * out_stride_ax + (size_t)i1 * out_stride_1 + (size_t)i2 * out_stride_2] = make_double2(sr, si);
  }
}

__global__ void real_to_complex_kernel(const double* __restrict__ f, double2* __restrict__ out, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    out[i] = make_double2(f[i], 0.0);
}

// F[G][G'] = |G| fhat(G - G') |G'| / (4 pi); fhat on the box [-m1..m1] x [-m2..m2] x [-m3..m3]
__global__ void fxc_matrix_kernel(DevSys d, const double2* __restrict__ fhat, int m1, int m2, int m3, double inv_nr,
                                  float2* __restrict__ F) {
  const int ng = d.ng0;
  const long long total = (long long)ng * ng;
  const double s4pi = 3.5449077018110318;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total; t += (long long)gridDim.x * blockDim.x) {
    const int g = (int)(t / ng), h = (int)(t - (long long)g * ng);
    const char4 a = d.gq[g], b = d.gq[h];
    const int dx = (int)a.x - (int)b.x + m1, dy = (int)a.y - (int)b.y + m2, dz = (int)a.z - (int)b.z + m3;
    const double2 v = fhat[((size_t)dx * (2 * m2 + 1) + dy) * (2 * m3 + 1) + dz];
    const float va = d.vsq[g], vb = d.vsq[h];
    float2 out = make_float2(0.f, 0.f);
    if (va > 0.f && vb > 0.f) {
      const double la = s4pi / va, lb = s4pi / vb;                // |G|, |G'|
      const double s = la * lb * inv_nr / (4.0 * 3.141592653589793);
      out = make_float2((float)(s * v.x), (float)(s * v.y));
    }
    F[t] = out;
  }
}

unsigned blocks_for(long long n, int threads) {
  long long b = (n + threads - 1) / threads;
  if (b > 152LL * 16) b = 152LL * 16;
  return (unsigned)(b < 1 ? 1 : b);
}

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace

size_t alda_ws_bytes(const DevSys& d) {
  const size_t nr = (size_t)d.n1 * d.n2 * d.n3;
  // f(r) (doubles), then two complex double buffers for the DFT passes (the first holds f as complex)
  return align256(nr * sizeof(double)) + 2 * align256(nr * sizeof(double2));
}

int launch_alda_kernel(const DevSys& d, const void* pair_ws, const int* m, void* F, void* ws, void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  const long long nr = (long long)d.n1 * d.n2 * d.n3;
  char* base = (char*)ws;
  double* f = (double*)base;
  double2* b0 = (double2*)(base + align256(nr * sizeof(double)));
  double2* b1 = (double2*)(base + align256(nr * sizeof(double)) + align256(nr * sizeof(double2)));
  alda_fxc_kernel<<<blocks_for(nr, 256), 256, 0, st>>>(d, (const float2*)pair_ws, f, 2.0 * d.norm);
  if (int e = (int)cudaGetLastError()) return e;
  real_to_complex_kernel<<<blocks_for(nr, 256), 256, 0, st>>>(f, b0, nr);
  if (int e = (int)cudaGetLastError()) return e;
  const int m1 = m[0], m2 = m[1], m3 = m[2];
  const int w1 = 2 * m1 + 1, w2 = 2 * m2 + 1, w3 = 2 * m3 + 1;
  // pass 1, x: b0 [x][y][z] -> b1 [j1][y][z]
  dft_pass_kernel<<<blocks_for((long long)w1 * d.n2 * d.n3, 128), 128, 0, st>>>(
      b0, b1, d.n1, m1, d.n2, d.n3, d.n2 * d.n3, d.n3, 1, d.n2 * d.n3, d.n3, 1);
  if (int e = (int)cudaGetLastError()) return e;
  // pass 2, y: b1 [j1][y][z] -> b0 [j1][j2][z]   (transformed axis y; other axes j1 (e1), z (e2))
  dft_pass_kernel<<<blocks_for((long long)w2 * w1 * d.n3, 128), 128, 0, st>>>(
      b1, b0, d.n2, m2, w1, d.n3, d.n3, d.n2 * d.n3, 1, d.n3, w2 * d.n3, 1);
  if (int e = (int)cudaGetLastError()) return e;
  // pass 3, z: b0 [j1][j2][z] -> b1 [j1][j2][j3]
  dft_pass_kernel<<<blocks_for((long long)w3 * w1 * w2, 128), 128, 0, st>>>(
      b0, b1, d.n3, m3, w1, w2, 1, w2 * d.n3, d.n3, 1, w2 * w3, w3);
  if (int e = (int)cudaGetLastError()) return e;
  fxc_matrix_kernel<<<blocks_for((long long)d.ng0 * d.ng0, 256), 256, 0, st>>>(d, b1, m1, m2, m3, 1.0 / (double)nr,
                                                                             (float2*)F);
  return (int)cudaGetLastError();
}

size_t epsm_ws_bytes(const DevSys& d, long long nw) {
  const size_t n = d.ng0;
  return align256((size_t)nw * n * (n + 1) * sizeof(float2)) + align256((size_t)nw * n * sizeof(float2));
}

int launch_epsilon_macro(const DevSys& d, const void* chi0, const void* F, int nw, void* eps_m, void* ws,
                         void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  const int n = d.ng0;
  char* base = (char*)ws;
  float2* aug = (float2*)base;
  float2* xb = (float2*)(base + align256((size_t)nw * n * (n + 1) * sizeof(float2)));
  if (F) {
    const long long rows = (long long)nw * n, step = 65535LL * gf::TM / n * n;      // whole frequencies per launch
    for (long long r = 0; r < rows; r += step) {
      const long long c = rows - r < step ? rows - r : step;
      kernel_rows_kernel<<<dim3((n + gf::TN - 1) / gf::TN, (unsigned)((c + gf::TM - 1) / gf::TM)), gf::kThreads, 0, st>>>(
          n, c, (const float2*)chi0 + (size_t)r * n, (const float2*)F, aug + (size_t)r * (n + 1));
      if (int e = (int)cudaGetLastError()) return e;
    }
  } else {
    augment_kernel<<<blocks_for((long long)nw * n * (n + 1), 256), 256, 0, st>>>(n, nw, (const float2*)chi0, aug);
    if (int e = (int)cudaGetLastError()) return e;
  }
  // the widest panel that leaves two CTAs an SM (n <= 433 for 16 columns, 842 for 8), down to 2 columns at n = 4096
  double2* out = (double2*)eps_m;
  if (solve_smem(n, 16) <= 112 * 1024) return launch_solve<16>(n, nw, aug, out, xb, st);
  if (solve_smem(n, 8) <= 112 * 1024) return launch_solve<8>(n, nw, aug, out, xb, st);
  if (solve_smem(n, 4) <= 200 * 1024) return launch_solve<4>(n, nw, aug, out, xb, st);
  return launch_solve<2>(n, nw, aug, out, xb, st);
}

}  // namespace bse
