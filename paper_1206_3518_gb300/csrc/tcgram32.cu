// Exchange part of H in FP32 accuracy on the tensor cores (step A3 of the FP32 build; Eq. V_eh):
//
//   H[S][S'] = sum_G conj(Y[S][G]) Y[S'][G] + delta_SS' (e_c + Delta - e_v),   Y[S][G] = rho_x[S][G] s(G),
//
// s(G) = sqrt(2 vbar(G) / (Omega Nk)), as FP16x3 products with promoted accumulation (tcf16.cuh) on the 128 x 128
// tiles (I <= J) of the upper triangle and the tiles (I, I - 1) just below it (a block of Nv Nc rows that
// straddles the row 128 I has upper entries there).  One image of Y serves both operands.
// Bound by the MMAs (0.70 of the sustained BF16 rate issued at dim 27648).  Measured with the split (ms; before: init_kernel on
// the FP32 pipes): fcc 4x4x4 3v3c 0.022 (0.030), fcc 8x8x8 3v4c 0.17 (1.65), fcc 12x12x12 4v4c 4.0 (53).
#include <cuda_runtime.h>

#include "internal.h"
#include "tcf16.cuh"

namespace bse {
namespace {

using tcf::kTileA;
using tcf::kTKC;
using tcf::kTM;

template <int GL, int NP>
__global__ __launch_bounds__(256) void split_y_kernel(DevSys d, const float2* __restrict__ rho_x,
                                                      unsigned char* __restrict__ img, float* __restrict__ inv, int nkc) {
  const int row = blockIdx.x * (256 / GL) + threadIdx.x / GL;
  const bool live = row < d.dim;
  const float2* x = rho_x + (size_t)(live ? row : 0) * d.ng_max;
  const float s = tcf::split_row<GL, NP>(x, d.ng0, d.xscale, img + (size_t)(row / kTM) * nkc * (2 * kTileA), 2 * kTileA,
                                         kTileA, row % kTM, live);
  if (live && threadIdx.x % GL == 0) inv[row] = s;
}

struct GramOp {
  static constexpr bool kReal = false, kConj = true, kHerm = false;
  int dim, nv, nc, nb, ng0, ntr, nkc;
  const unsigned char* img;
  const float* inv;
  const double* e;
  double delta;
  float2* H;
  int* status;
  long long nupper, ntiles;                     // tiles I <= J, row by row; then (I, I - 1)

  __device__ __forceinline__ long long row_start(int I) const { return (long long)I * ntr - (long long)I * (I - 1) / 2; }
  __device__ __forceinline__ bool tile(long long t, tcf::Tile& o) const {
    int I, J;
    if (t >= nupper) {
      I = (int)(t - nupper) + 1;
      J = I - 1;
    } else {
      const double b = 2.0 * ntr + 1.0;
      I = (int)floor(0.5 * (b - sqrt(fmax(b * b - 8.0 * (double)t, 0.0))));
      I = I < 0 ? 0 : (I > ntr - 1 ? ntr - 1 : I);
      while (I > 0 && row_start(I) > t) --I;
      while (I + 1 < ntr && row_start(I + 1) <= t) ++I;
      J = I + (int)(t - row_start(I));
    }
    o.a = img + (size_t)I * nkc * (2 * kTileA);
    o.b = img + (size_t)J * nkc * (2 * kTileA);
    o.a_step = o.b_step = 2 * kTileA;
    o.K = ng0;
    o.n = kTM;
    o.m0 = I * kTM;
    o.n0 = J * kTM;
    o.mvalid = dim - o.m0;
    o.nvalid = min(kTM, dim - o.n0);
    o.batch = 0;
    o.row0 = o.m0;
    return true;
  }
  __device__ __forceinline__ float2* row_out(const tcf::Tile& t, int row) const {
    return H + (size_t)(t.m0 + row) * dim + t.n0;
  }
  __device__ __forceinline__ float row_scale(const tcf::Tile& t, int row) const { return inv[t.m0 + row]; }
  __device__ __forceinline__ float col_scale(const tcf::Tile& t, int col) const { return inv[t.n0 + col]; }
  __device__ __forceinline__ float2 value(const tcf::Tile& t, int row, int col, float2 s) const {
    const int S = t.m0 + row;
    if (S == t.n0 + col) {
      const int ic = S % nc, iv = (S / nc) % nv, k = S / (nv * nc);
      s.x += (float)(e[(size_t)k * nb + nv + ic] + delta - e[(size_t)k * nb + iv]);
    }
    return s;
  }
};

size_t img_bytes(const DevSys& d) {
  return (size_t)((d.dim + kTM - 1) / kTM) * ((d.ng0 + kTKC - 1) / kTKC) * (2 * kTileA);
}

template <int GL, int NP>
void launch_split(const DevSys& d, const void* rho_x, unsigned char* img, float* inv, int nkc, cudaStream_t st) {
  constexpr int rows = 256 / GL;
  split_y_kernel<GL, NP><<<(unsigned)((d.dim + rows - 1) / rows), 256, 0, st>>>(d, (const float2*)rho_x, img, inv, nkc);
}

}  // namespace

size_t gram32_ws_bytes(const DevSys& d) { return kWsSlack + img_bytes(d) + (((size_t)d.dim * sizeof(float) + 255) & ~(size_t)255); }

int launch_kernel_init_tc32(const DevSys& d, const void* rho_x, const double* energies, double delta, void* H, void* ws,
                            int* status, void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  unsigned char* img = ws_base(ws);
  float* inv = (float*)(img + img_bytes(d));
  const int nkc = (d.ng0 + kTKC - 1) / kTKC;
  if (nkc < 1) return (int)cudaErrorInvalidValue;
  if (d.ng0 <= 128)
    launch_split<16, 1>(d, rho_x, img, inv, nkc, st);
  else if (d.ng0 <= 384)
    launch_split<16, 3>(d, rho_x, img, inv, nkc, st);
  else
    launch_split<32, 3>(d, rho_x, img, inv, nkc, st);
  if (int e = (int)cudaGetLastError()) return e;
  GramOp op;
  op.dim = d.dim;
  op.nv = d.nv;
  op.nc = d.nc;
  op.nb = d.nb;
  op.ng0 = d.ng0;
  op.ntr = (d.dim + kTM - 1) / kTM;
  op.nkc = nkc;
  op.img = img;
  op.inv = inv;
  op.e = energies;
  op.delta = delta;
  op.H = (float2*)H;
  op.status = status;
  op.nupper = (long long)op.ntr * (op.ntr + 1) / 2;
  op.ntiles = op.nupper + op.ntr - 1;
  return tcf::launch(op, stream);
}

}  // namespace bse
