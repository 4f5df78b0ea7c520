// Direct pair densities on the 5th-generation tensor cores (step A2 of the mixed build, and of the FP32 build where
// tcpair_preferred says so; Eq. pair_density in the plane-wave basis):
//
//   rho_nm^{kk'}(G) = sum_{G2 in S(k')} conj(c_nk(G2 - G)) c_mk'(G2),   G = g_p(q) - G0.
//
// For a fixed k the factor conj(c_nk(G2 - G)), a function of (G, G2), is the same for every block
// (k, k').  The blocks of one k whose k' lie in one region of the k' mesh (the plan's regions: a few
// neighbouring mesh points) therefore form one GEMM per band n of the set (vv' or cc'):
//
//   D[G][(k', m)] = sum_{G2 in K} A_n[G][G2] B[(k', m)][G2],
//
//   rows G     the union over the tile's blocks of the G sphere of their q (shifted by G0): the first
//              block's sphere in its sphere order, then the other points in lexicographic order;
//   K          the region's layout, the union of the spheres S(k') of its points;
//   columns    the tile's blocks times the bands m of the set.
//
// A_n is gathered from a dense difference box in shared memory that holds the coefficients of band n themselves
// (zero off S(k)): one 8-byte lookup per element.  B comes from packed panels of the coefficients of each
// region's points in its K layout (zero off S(k')), written once per call.  The epilogue keeps, for every block,
// the rows on its own sphere and writes them at their sphere positions, so the output is the direct set of
// the correlation kernels.
//
// Arithmetic (FP16x3, tcf16.cuh): the coefficients of every (k, band) are scaled by a power of two and split
// hi + lo in FP16 (22 bits); each real product is hi.lo + lo.hi + hi.hi, and the tensor core's accumulator holds
// one K chunk (SUB panels of 32 complex values, tp_fit) at a time, which the epilogue warps add to FP32
// registers.  The result has the accuracy of the FP32 correlation kernel, so one kernel serves both precisions of the build.  The G = 0 overlaps
// of the diagonal blocks (k' = k), which meet the q = 0 head of W, are summed again in FP64
// afterwards (tcpair_diag_kernel).
//
// tcpair_kernel is persistent (one CTA per SM); its CTAs deal the tiles (k, region) among themselves (deal_tiles); a pass
// is one band n and 128 rows.  Four warpgroups share the registers (setmaxnreg):
//   0, 1  promote the chunks of the even / odd passes into registers and write the pass's densities while the
//         other group promotes the next pass (the scattered 8-byte stores, one cache line each, take most of
//         a pass);
//   2     gathers the A tile of each K chunk straight into tensor memory (4 / SUB slots, tcgen05.st);
//   3     two warps issue the MMAs (12 per 16 complex K, A from tensor memory, B from shared memory; warp-uniform,
//         umma.cuh), one warp brings the B rows into a ring of shared-memory stages with bulk copies (the region's
//         panels of the chunk: hi rows and lo rows); the columns of a region's points without a block in
//         the tile are computed and dropped.
// At most 64 columns per pass: a group's sums are 2 x 64 registers a thread, and two accumulators (Re | Im, 128 TMEM
// columns each) and four A slots fill tensor memory.  Every mbarrier wait is bounded (2 s); on expiry the CTA records
// BSE_ERR_TIMEOUT, stops issuing, waits (bounded) for its MMAs in flight, frees its tensor memory and returns.
//
// What bounds it: no single part.  With a ring of two stages (fcc 8x8x8 3v4c 10.9 ms; fcc 12x12x12 4v4c, 144 q 45.8) a copy
// without the tensor-memory stores of A takes 8.0 and 35.2 ms, without the lookups 8.7 and 40.5, without the stores of
// the densities 9.5 and 39.4, with a twelfth of the MMAs 9.0 and 35.7, without the promotion 10.8 and 44.9: the gather's stores meet the
// accumulators' traffic in tensor memory (the MMAs take 960 of ~1600 cycles per 32 K).  On sheets (K of 160) the
// set-up of a tile is as long as its passes.  Measured (ms; before: the FP32 correlation kernel / BF16x3 tensor kernel with 96
// columns, two lookups an element and one accumulator a pass): fcc 8x8x8 3v4c 9.7 (50.1 / 15.2), fcc 12x12x12 4v4c,
// q 144 to 288 43.2 (363 / 59), 27x27 sheet 2v3c, 64 q 0.96 (1.52 / -).  Error against 64 bits (2-norm of random states'
// densities, nine systems from 3 to 12 Ha): 1.7e-7 to 2.1e-7 (correlation kernel 1.6e-7 to 5.5e-7, growing with the
// sphere; below it only at 5x5x5 4v4c, 3 Ha: 1.6e-7 against 1.8e-7).
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "internal.h"
#include "tcf16.cuh"
#include "umma.cuh"

namespace bse {
namespace {

using umma::mbar_arrive;
using umma::mbar_init;
using umma::mbar_wait;
using umma::mma_commit;
using umma::smem_u32;
using umma::swz;

constexpr int kGroups = 2;                     // epilogue warpgroups (warps 0-3, 4-7)
constexpr int kG0 = 8, kGWarps = 4;            // gather warpgroup
constexpr int kMmaWarp = 12, kB0 = 14;         // two MMA issue warps, B producer (bulk copies)
constexpr int kThreads = 512;
// 128 registers a thread at launch; 168 + 168 + 112 + 64 = 4 x 128
constexpr int kRegEpi = 168, kRegGather = 112, kRegIssue = 64;
constexpr int kMaxStages = 6;                  // B ring depth at most, in panels of 32 complex K
constexpr int kASlots = 4;                     // A tiles of 32 complex K in tensor memory
constexpr int kGThreads = kGWarps * 32;
constexpr int kNCols = 64;                     // columns (k', band) of a pass at most
constexpr int kAcc = 2 * kNCols;               // one accumulator: Re [0, 64), Im [64, 128)
constexpr int kTKC = 32;                       // complex K values of a packed panel
constexpr int kACols = 64;                     // one A tile in TMEM: two K16 halves x (Re hi, Im hi, Re lo, Im lo) x 8
constexpr int kImgRow = 256;                   // packed image of 32 K values: hi row (128 B), lo row (128 B)
size_t align16(size_t x) { return (x + 15) & ~(size_t)15; }

struct TpGeo {
  int q_begin, nqc;
  int table;                                    // the list of differences has room in the ring (deal_tiles)
  int share;                                    // which kMine kThreads tiles of every CTA's share the launch takes
  long long vbase;
  int nkc;                                      // K panels of the packed images (tc_kpad / 32)
  int sub;                                      // panels per stage (a promoted chunk): 1 or 2
  int stages, nmax;                             // ring depth; B rows per stage (max columns, multiple of 16)
  int cap;                                      // rows of the position table
  int sub_bytes, stage_bytes;                   // a panel's B rows; a stage's
  int by, bz, box_n, box_c;                     // difference box of S(k): dims, entries, key of G1 = 0
  int rowbox, nwords, wpl;                      // row box: entries, bit words, words per (x, y) line
  int o_bar, o_box, o_pkey, o_kkey, o_rows, o_bits, o_slot, o_binfo, o_bptr, o_binv, o_ptab;
  size_t smem;                                  // dynamic shared memory incl. 1 KB alignment slack
};

TpGeo tp_geo(const DevSys& d, int sub, int stages, int cap) {
  TpGeo g{};
  g.sub = sub;
  g.stages = stages;
  g.cap = cap;
  g.nkc = d.tc_kpad / kTKC;
  const int mb = d.nv > d.nc ? d.nv : d.nc;
  g.nmax = (d.tc_rsize * mb + 15) / 16 * 16;
  g.sub_bytes = 2 * g.nmax * umma::kRow;        // B hi rows, B lo rows
  g.stage_bytes = sub * g.sub_bytes;
  const int rx = d.fwf[0] + d.fpair[0], ry = d.fwf[1] + d.fpair[1], rz = d.fwf[2] + d.fpair[2];
  g.by = 2 * ry + 1;
  g.bz = 2 * rz + 1;
  g.box_n = (2 * rx + 1) * g.by * g.bz;
  g.box_c = (rx * g.by + ry) * g.bz + rz;
  g.rowbox = (2 * d.fpair[0] + 1) * (2 * d.fpair[1] + 1) * (2 * d.fpair[2] + 1);
  g.wpl = (2 * d.fpair[2] + 1 + 31) / 32;
  g.nwords = (2 * d.fpair[0] + 1) * (2 * d.fpair[1] + 1) * g.wpl;
  size_t o = (size_t)stages * g.stage_bytes;
  g.o_bar = (int)o; o += align16((size_t)(2 * stages + 2 * (kASlots / sub) + 2 * kGroups + 4) * 8 + 8 * sizeof(int));
  g.o_box = (int)o; o += align16((size_t)g.box_n * 8);
  g.o_pkey = (int)o; o += align16((size_t)d.npw_max * 4);
  g.o_kkey = (int)o; o += align16((size_t)d.tc_kpad * 4);
  g.o_rows = (int)o; o += align16((size_t)g.rowbox * 4);
  g.o_bits = (int)o; o += align16((size_t)g.nwords * 4);
  g.o_slot = (int)o; o += align16((size_t)d.tc_rsize * 4);
  g.o_binfo = (int)o; o += align16((size_t)d.tc_rsize * 16);
  g.o_bptr = (int)o; o += align16((size_t)d.tc_rsize * 16);
  g.o_binv = (int)o; o += align16((size_t)d.tc_rsize * d.nb * 4);
  g.o_ptab = (int)o; o += align16((size_t)cap * d.tc_rsize * 2);
  g.smem = o + 1024;
  return g;
}

__device__ __forceinline__ void fail_now(volatile int* fail, int* status) {
  *fail = 1;
  atomicCAS(status, 0, (int)BSE_ERR_TIMEOUT);
}

__device__ __forceinline__ void gather_bar() { asm volatile("barrier.sync 1, %0;" ::"n"(kGThreads) : "memory"); }

__device__ __forceinline__ uint2 lds64(uint32_t addr) {
  uint2 v;
  asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr));
  return v;
}

// x = hi + lo in FP16 as (hi | lo << 16)
__device__ __forceinline__ uint32_t split_word(float x) {
  const __half h = __float2half_rn(x);
  const __half l = __float2half_rn(x - __half2float(h));
  return (uint32_t)__half_as_ushort(h) | ((uint32_t)__half_as_ushort(l) << 16);
}

// ---------------------------------------------------------------- packed coefficient panels
// Packed B panels: for each region r, set (valence bands, then conduction bands) and K chunk c, the rows
// j = slot nset + m of every k' of the region (slot: its position in the region, m: its band in the set),
// [Re 32 | Im 32] FP16 in the region's K layout (zero off S(k')), hi rows then lo rows, the 16-byte chunks of
// row j permuted by j mod 8 (128B swizzle): a stage's B tile is two bulk copies.
__device__ __forceinline__ size_t panel_off(const DevSys& d, int r, int set, int c, int nkc) {
  const size_t per_r = (size_t)nkc * 2 * umma::kRow * d.tc_rsize * (d.nv + d.nc);
  const size_t set_off = set ? (size_t)nkc * 2 * umma::kRow * d.tc_rsize * d.nv : 0;
  const int nset = set ? d.nc : d.nv;
  return (size_t)r * per_r + set_off + (size_t)c * 2 * umma::kRow * d.tc_rsize * nset;
}

__device__ __forceinline__ void region_of(const DevSys& d, int k2, int& r, int& slot) {
  const int o0 = k2 / (d.nk2 * d.nk3), o1 = (k2 / d.nk3) % d.nk2, o2 = k2 % d.nk3;
  r = ((o0 / d.tc_rg[0]) * d.tc_nr[1] + o1 / d.tc_rg[1]) * d.tc_nr[2] + o2 / d.tc_rg[2];
  slot = ((o0 % d.tc_rg[0]) * d.tc_rg[1] + o1 % d.tc_rg[1]) * d.tc_rg[2] + o2 % d.tc_rg[2];
}

// scale[k nb + band]: the power of two that puts the largest component of c_{k,band} into [2^14, 2^15); its inverse
// in the second half.  One warp per (k, band): the plain copy of the coefficients (the other densities read it), their
// scale, the row's panels zeroed and its sphere points written.  Part of the real-space stage where the route is the
// default (tcpair_packed), so that the direct stages only read the workspace and a set of q chunks packs once.
__global__ __launch_bounds__(256) void tcpair_pack_kernel(DevSys d, const float2* __restrict__ coef,
                                                          float2* __restrict__ copy, float* __restrict__ scale,
                                                          unsigned char* __restrict__ bimg, int nkc) {
  const int row = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;   // k nb + band
  if (row >= d.nkpt * d.nb) return;
  const int k = row / d.nb, band = row - k * d.nb, n = d.npw[k];
  const float2* x = coef + (size_t)row * d.npw_max;
  float2* y = copy ? copy + (size_t)row * d.npw_max : nullptr;
  float m = 0.f;
#pragma unroll 4
  for (int i = lane; i < d.npw_max; i += 32) {
    const float2 c = x[i];
    if (copy) y[i] = c;
    if (i < n) m = fmaxf(m, fmaxf(fabsf(c.x), fabsf(c.y)));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  const int e = tcf::scale_exp(m);
  const float sc = tcf::pow2(e);
  if (lane == 0) {
    scale[row] = sc;
    scale[d.nkpt * d.nb + row] = tcf::pow2(-e);
  }
  const int set = band < d.nv ? 0 : 1, nset = set ? d.nc : d.nv;
  int r, slot;
  region_of(d, k, r, slot);
  const int j = slot * nset + (set ? band - d.nv : band), ph = j & 7;
  const size_t lo_off = (size_t)d.tc_rsize * nset * umma::kRow;
  unsigned char* img = bimg + panel_off(d, r, set, 0, nkc) + (size_t)j * umma::kRow;   // chunk c: + 2 c lo_off
  for (int t = lane; t < nkc * 16; t += 32)     // 2 x 128 bytes per chunk
    *reinterpret_cast<uint4*>(img + (size_t)(t >> 3) * lo_off + (t & 7) * 16) = make_uint4(0u, 0u, 0u, 0u);
  __syncwarp();
  const short* kpos = d.tc_kpos + (size_t)k * d.npw_max;
#pragma unroll 4
  for (int i = lane; i < n; i += 32) {
    const int l = kpos[i], at = l % kTKC;
    const float2 c = x[i];
    const uint32_t re = split_word(c.x * sc), im = split_word(c.y * sc);
    unsigned short* hi = reinterpret_cast<unsigned short*>(img + (size_t)(2 * (l / kTKC)) * lo_off);
    unsigned short* lo = reinterpret_cast<unsigned short*>(reinterpret_cast<unsigned char*>(hi) + lo_off);
    const int cr = ((at >> 3) ^ ph) * 8 + (at & 7), ci = ((4 + (at >> 3)) ^ ph) * 8 + (at & 7);
    hi[cr] = (unsigned short)(re & 0xFFFFu);
    hi[ci] = (unsigned short)(im & 0xFFFFu);
    lo[cr] = (unsigned short)(re >> 16);
    lo[ci] = (unsigned short)(im >> 16);
  }
}

// ---------------------------------------------------------------- tiles of a q range
// A tile is a region and a k.  It has a block where some k' of the region has q = k' - k in the range and k <= k'; whether
// the first holds depends on the difference of the region's corner and k alone.  The CTAs list the differences that do
// and deal the tiles (region, difference) among themselves, the i-th one to CTA i mod grid, from the plan's tables
// alone: a call keeps nothing in the workspace, so calls that share it may overlap.  Regions in order: the CTAs in
// flight share one region's packed B rows, which stay in L2.  The tiles of the most passes are dealt first, so that every
// CTA gets as many of each kind (dealt by the fullness of the region a sheet's chunk took up to 10% longer).
struct Point {                                   // offsets on the mesh
  int x, y, z;
};
__device__ __forceinline__ int wrap(int x, int n) { return x < 0 ? x + n : x >= n ? x - n : x; }
__device__ __forceinline__ int index_of(const DevSys& d, Point p) { return (p.x * d.nk2 + p.y) * d.nk3 + p.z; }
__device__ __forceinline__ Point point_of(const DevSys& d, int i) {
  return {i / (d.nk2 * d.nk3), (i / d.nk3) % d.nk2, i % d.nk3};
}
__device__ __forceinline__ Point plus(const DevSys& d, Point a, Point b) {
  return {wrap(a.x + b.x, d.nk1), wrap(a.y + b.y, d.nk2), wrap(a.z + b.z, d.nk3)};
}
__device__ __forceinline__ Point minus(const DevSys& d, Point a, Point b) {
  return {wrap(a.x - b.x, d.nk1), wrap(a.y - b.y, d.nk2), wrap(a.z - b.z, d.nk3)};
}
__device__ __forceinline__ Point corner_of(const DevSys& d, int r) {
  return {r / (d.tc_nr[1] * d.tc_nr[2]) * d.tc_rg[0], (r / d.tc_nr[2]) % d.tc_nr[1] * d.tc_rg[1],
          r % d.tc_nr[2] * d.tc_rg[2]};
}
// Block in the q range of k and the slot's point, given the difference of the region's corner and k; -1: none.
__device__ __forceinline__ int block_of(const DevSys& d, const TpGeo& g, int k, Point diff, int s) {
  const Point o = {s / (d.tc_rg[1] * d.tc_rg[2]), (s / d.tc_rg[2]) % d.tc_rg[1], s % d.tc_rg[2]};
  const int q = index_of(d, plus(d, diff, o));
  return q >= g.q_begin && q < g.q_begin + g.nqc ? d.blkidx[(size_t)q * d.nkpt + k] : -1;
}
// Points of a box of (e0, e1, e2) at difference p whose own difference lies in the q range: runs along the last axis that
// has more than one point, each one or two intervals of q.
__device__ __forceinline__ int near_points(const DevSys& d, const TpGeo& g, Point p, int e0, int e1, int e2) {
  if (g.nqc == d.nkpt) return e0 * e1 * e2;
  const bool z = d.nk3 > 1;
  const int len = z ? e2 : e1, nl = z ? d.nk3 : d.nk2, at = z ? p.z : p.y, rows = z ? e1 : 1;
  const int qe = g.q_begin + g.nqc;
  int m = 0;
  for (int a = 0; a < e0; ++a)
    for (int b = 0; b < rows; ++b) {
      const int x = wrap(p.x + a, d.nk1), base = z ? (x * d.nk2 + wrap(p.y + b, d.nk2)) * d.nk3 : x * d.nk2;
      m += max(0, min(qe, base + min(at + len, nl)) - max(g.q_begin, base + at));
      m += max(0, min(qe, base + at + len - nl) - max(g.q_begin, base));
    }
  return m;
}

// Class of the tiles of difference p, the most passes first; -1: no point in the range.  The passes of a tile follow from
// the rows of its blocks, those of the layers of the region that are at least half in the range (whole layers are in the
// plan's table; a range cuts a layer at its ends only).
constexpr int kMine = 2, kFill = 4;              // list entries per thread; classes
__device__ __forceinline__ int class_of(const DevSys& d, const TpGeo& g, Point p) {
  const bool ax = d.tc_axis == 0;
  const int e0 = ax ? 1 : d.tc_rg[0], e1 = ax ? d.tc_rg[1] : 1, e2 = d.tc_rg[2], half = (e0 * e1 * e2 + 1) / 2;
  int first = -1, last = -1, any = -1;
  if (g.nqc == d.nkpt) {
    first = 0;
    last = any = d.tc_layers - 1;
  } else if (!ax && d.nk3 == 1) {                // layers of one point: a run along axis 1 and its part beyond the mesh's end
    const int base = p.x * d.nk2, end = p.y + d.tc_layers - d.nk2, qe = g.q_begin + g.nqc;
    const int lo = max(g.q_begin - base, p.y), hi = min(qe - base, min(p.y + d.tc_layers, d.nk2));
    const int lo2 = max(g.q_begin - base, 0), hi2 = min(qe - base, end);
    if (hi > lo) {
      first = lo - p.y;
      last = hi - 1 - p.y;
    }
    if (hi2 > lo2) {
      first = first < 0 ? lo2 + d.nk2 - p.y : first;
      last = hi2 - 1 + d.nk2 - p.y;
    }
    any = last;
  } else {
    for (int l = 0; l < d.tc_layers; ++l) {
      const int m = near_points(d, g, plus(d, p, ax ? Point{l, 0, 0} : Point{0, l, 0}), e0, e1, e2);
      if (m >= half) {
        first = first < 0 ? l : first;
        last = l;
      }
      if (m > 0) any = l;
    }
  }
  if (any < 0) return -1;
  if (first < 0) first = last = any;
  const int at = index_of(d, plus(d, p, ax ? Point{first, 0, 0} : Point{0, first, 0}));
  return min(kFill - 1, d.tc_maxpass - (int)d.tc_passes[(size_t)at * d.tc_layers + last - first]);
}

// Tiles of this CTA (its share of the launch) as region nkpt + k in the first kList words of scratch; returns their
// number.  (Not inlined: its registers are not those of the passes.)  After the list: sums of the warps, differences (without
// room for them every difference of the mesh is tried).  Where k lies within the region only some of its points come after
// k: such tiles are dealt last, and next_tile passes over one without a block.
constexpr int kList = kMine * kThreads, kDealSums = kFill * (kThreads / 32);
__device__ __noinline__ int deal_tiles(const DevSys& d, const TpGeo& g, int* scratch) {
  constexpr int kWarps = kThreads / 32;
  int* list = scratch;
  int* sums = list + kList;                      // [class][warp]
  unsigned* diffs = (unsigned*)(sums + kDealSums);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // exclusive prefix over the threads of n[class], classes in order; returns the total
  auto prefix = [&](int (&n)[kFill], int (&start)[kFill + 1]) {
    int incl[kFill];
#pragma unroll
    for (int f = 0; f < kFill; ++f) {
      incl[f] = n[f];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, incl[f], o);
        if (lane >= o) incl[f] += u;
      }
      if (lane == 31) sums[f * kWarps + warp] = incl[f];
    }
    __syncthreads();
    start[0] = 0;
#pragma unroll
    for (int f = 0; f < kFill; ++f) {
      int before = 0, all = 0;
      for (int i = 0; i < kWarps; ++i) {
        const int u = sums[f * kWarps + i];
        before += i < warp ? u : 0;
        all += u;
      }
      n[f] = start[f] + before + incl[f] - n[f];
      start[f + 1] = start[f] + all;
    }
    __syncthreads();
  };

  // the differences with a point in the range, by class
  const int per_d = (d.nkpt + kThreads - 1) / kThreads, d0 = min(tid * per_d, d.nkpt), d1 = min(d0 + per_d, d.nkpt);
  int n[kFill], start[kFill + 1];
#pragma unroll
  for (int f = 0; f < kFill; ++f) n[f] = 0;
  for (int i = d0; i < d1; ++i) {
    const int cls = class_of(d, g, point_of(d, i));
#pragma unroll
    for (int f = 0; f < kFill; ++f) n[f] += cls == f ? 1 : 0;
  }
  prefix(n, start);
  const bool table = g.table != 0;
  if (table) {
    for (int i = d0; i < d1; ++i) {
      const Point p = point_of(d, i);
      const int cls = class_of(d, g, p);
#pragma unroll
      for (int f = 0; f < kFill; ++f)
        if (cls == f) diffs[n[f]++] = (unsigned)(p.x | p.y << 10 | p.z << 20);
    }
    __syncthreads();
  } else {                                       // one class of all differences
#pragma unroll
    for (int f = 0; f < kFill; ++f) start[f + 1] = d.nkpt;
  }

  // candidate tiles: class, region, difference
  const long long cand = (long long)d.tc_nreg * start[kFill], per = (cand + kThreads - 1) / kThreads;
  const long long i0 = min(tid * per, cand), i1 = min(i0 + per, cand);
  auto scan = [&](auto&& live) {
    int f = 0;
    while (f < kFill - 1 && i0 >= (long long)d.tc_nreg * start[f + 1]) ++f;
    int size = start[f + 1] - start[f];
    const long long in = i0 - (long long)d.tc_nreg * start[f];
    int r = size > 0 ? (int)(in / size) : 0, j = (int)(in - (long long)r * size);
    Point c = corner_of(d, r);
    for (long long i = i0; i < i1; ++i) {
      while (j >= size) {                        // next region, or the next class with any difference
        j = 0;
        if (size > 0 && ++r < d.tc_nreg) {
          c = corner_of(d, r);
          break;
        }
        r = 0;
        c = corner_of(d, 0);
        ++f;
        size = start[f + 1] - start[f];
      }
      const int at = start[f] + j++;
      const unsigned w = table ? diffs[at] : 0u;
      const Point diff = table ? Point{(int)(w & 1023u), (int)((w >> 10) & 1023u), (int)(w >> 20)} : point_of(d, at);
      const int k = index_of(d, minus(d, c, diff));
      bool any = k <= index_of(d, {c.x + d.tc_rg[0] - 1, c.y + d.tc_rg[1] - 1, c.z + d.tc_rg[2] - 1});
      if (any && d.nfill > 0) {                  // representatives only: look the blocks up
        any = false;
        for (int s = 0; s < d.tc_rsize && !any; ++s) any = block_of(d, g, k, diff, s) >= 0;
      }
      if (any) live(r, k, k > index_of(d, c) ? 1 : 0);
    }
  };
#pragma unroll
  for (int f = 0; f < kFill; ++f) n[f] = 0;
  if (i0 < i1) scan([&](int, int, int part) { part ? ++n[1] : ++n[0]; });
  const bool some = n[0] + n[1] > 0;
  int total[kFill + 1];
  prefix(n, total);                              // the tiles with k within the region (part) after all others
  const int grid = (int)gridDim.x, own = (int)blockIdx.x, all = total[kFill], e0 = g.share * kList;
  if (some)
    scan([&](int r, int k, int part) {
      const int rank = part ? n[1]++ : n[0]++, e = rank / grid;
      if (rank - e * grid == own && e >= e0 && e < e0 + kList) list[e - e0] = r * d.nkpt + k;
    });
  __syncthreads();
  return all > own ? min(kList, max(0, (all - 1 - own) / grid + 1 - e0)) : 0;
}

// ---------------------------------------------------------------- the GEMM tiles
// One row of a pass to its blocks: NSET columns per slot, unrolled (a loop over columns with the slot's tables and
// branches in it took as long as the promotion of the pass; where the stores go makes no difference: consecutive
// addresses instead of sphere positions measured the same).  SMALL: the row's inverse scale is below 1 and is taken first,
// else last, so that no product leaves FP32's range that the result does not leave (the smaller of the two first, chosen
// per column, took 1% of the build).
template <int NSET, bool SMALL>
__device__ __forceinline__ void write_pass(const float (&re)[kNCols], const float (&im)[kNCols], float ia,
                                           const float* ib, float2* const* bptr, const short* pt, int rs, int nb,
                                           size_t first, int ng_max) {
#pragma unroll
  for (int b = 0; b < kNCols / NSET; ++b) {
    if (b >= rs) break;
    const int pb = pt[b];
    float2* dst = bptr[2 * b] + first + pb;
#pragma unroll
    for (int m = 0; m < NSET; ++m) {
      const float s = ib[b * nb + m], x = SMALL ? ia : s, y = SMALL ? s : ia;
      const float2 v = make_float2(re[b * NSET + m] * x * y, im[b * NSET + m] * x * y);
      if (pb >= 0) dst[(size_t)m * ng_max] = v;
    }
  }
}

template <int SUB>
__global__ __launch_bounds__(kThreads, 1) void tcpair_kernel(const __grid_constant__ DevSys d, const float2* __restrict__ coef,
                                                             const float* __restrict__ scale,
                                                             const unsigned char* __restrict__ bimg,
                                                             float2* __restrict__ out,
                                                             const __grid_constant__ TpGeo g, int* status) {
  constexpr int kAStages = kASlots / SUB, kACols_ = SUB * kACols, kChunk = SUB * kTKC;
  extern __shared__ __align__(1024) unsigned char tp_smem_raw[];
  unsigned char* sm = (unsigned char*)(((uintptr_t)tp_smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full_b = (uint64_t*)(sm + g.o_bar);   // [stages] B rows landed
  uint64_t* empty_b = full_b + g.stages;          // [stages] MMAs done with the B stage
  uint64_t* full_a = empty_b + g.stages;          // [slots] A tile written to tensor memory
  uint64_t* empty_a = full_a + kAStages;          // [slots] MMAs done with the A tile
  uint64_t* tfull = empty_a + kAStages;           // [group][2] accumulator holds a chunk of one of the group's passes
  uint64_t* tempty = tfull + 2 * kGroups;          // [2] accumulator promoted
  uint64_t* drain = tempty + 2;                    // [2] every MMA of an issue warp complete
  int* iv = (int*)(drain + 2);                     // tmem, fail, tile, rows, points in the box, last tile with a block
  volatile int* fail = iv + 1;
  uint2* box = (uint2*)(sm + g.o_box);
  int* pkey = (int*)(sm + g.o_pkey);
  int* kkey = (int*)(sm + g.o_kkey);
  char4* rows = (char4*)(sm + g.o_rows);
  unsigned* bits = (unsigned*)(sm + g.o_bits);
  int* slot = (int*)(sm + g.o_slot);
  int4* binfo = (int4*)(sm + g.o_binfo);
  float2** bptr = (float2**)(sm + g.o_bptr);       // [slot][set] first vector of the block
  float* binv = (float*)(sm + g.o_binv);           // [slot][band] inverse scale of the point's coefficients
  short* ptab = (short*)(sm + g.o_ptab);           // [row][slot] sphere position of the row on the slot's block, or -1

  const int tid = threadIdx.x, warp = umma::uniform(tid >> 5), lane = tid & 31;
  const int rs = d.tc_rsize;
  const int f0 = d.fwf[0], f1 = d.fwf[1], f2 = d.fwf[2];
  const int kb1 = 2 * f1 + 1, kb2 = 2 * f2 + 1;
  const int p0 = d.fpair[0], p1 = d.fpair[1], p2 = d.fpair[2];
  const int rb1 = 2 * p1 + 1;
  const int nv = d.nv, nc = d.nc, nb = d.nb;
  constexpr uint32_t a_col0 = 2 * kAcc;            // the A slots after the two accumulators

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(iv)), "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 32) {
    for (int i = 0; i < g.stages; ++i) {
      mbar_init(smem_u32(full_b + i), 1);
      mbar_init(smem_u32(empty_b + i), 1);
    }
    for (int i = 0; i < kAStages; ++i) {
      mbar_init(smem_u32(full_a + i), kGWarps);
      mbar_init(smem_u32(empty_a + i), 1);
    }
    for (int i = 0; i < 2 * kGroups; ++i) mbar_init(smem_u32(tfull + i), 1);
    for (int i = 0; i < 2; ++i) mbar_init(smem_u32(tempty + i), 4);
    for (int i = 0; i < 2; ++i) mbar_init(smem_u32(drain + i), 1);
    iv[1] = 0;
    iv[4] = 0;
    iv[5] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int i = tid; i < g.box_n; i += kThreads) box[i] = make_uint2(0u, 0u);
  const int nmine = deal_tiles(d, g, (int*)sm);  // (the ring is not in use yet)
  int mine[kMine];                               // entry e: mine[e / kThreads] of thread e % kThreads
#pragma unroll
  for (int i = 0; i < kMine; ++i) mine[i] = ((const int*)sm)[i * kThreads + tid];   // (past the number: not used)
  asm volatile("fence.proxy.async;" ::: "memory");   // bulk copies write the ring next
  int taken = 0;
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = umma::uniform((uint32_t)iv[0]);

  const int role = warp >> 2;                    // 0, 1 epilogue, 2 gather, 3 issue
  unsigned sc = 0, pc = 0;                       // stages and passes issued so far (the same in every role)
  int r = 0, k = 0, kc = 0, MT = 0, nmt = 0, nch = 0, n1 = 0;

  const size_t pq = (size_t)(2 * f0 + 1) * kb1 * kb2;
  auto position = [&](char4 G, int4 bi) -> short {
    const int x = G.x + (bi.z & 3) - 1, y = G.y + ((bi.z >> 2) & 3) - 1, z = G.z + ((bi.z >> 4) & 3) - 1;
    if (bi.x < 0 || x < -f0 || x > f0 || y < -f1 || y > f1 || z < -f2 || z > f2) return -1;
    return d.tc_pmap[(size_t)bi.x * pq + ((size_t)(x + f0) * kb1 + y + f1) * kb2 + z + f2];
  };

  // The next tile and its tables (all 512 threads, each role from its own copy of the tile loop: the register split
  // only holds where the roles' code does not meet).  False: no tile is left.
  auto all_bar = []() { asm volatile("barrier.sync 2, %0;" ::"n"(kThreads) : "memory"); };
  auto next_tile = [&]() -> bool {
    sc += (unsigned)(nb * nmt * nch);
    pc += (unsigned)(nb * nmt);
    do {                                         // (a tile dealt may turn out to have no block)
      all_bar();                                 // every role is done with the previous tile
      if (tid == taken % kThreads) iv[2] = *fail || taken >= nmine ? -1 : taken < kThreads ? mine[0] : mine[1];
      ++taken;
      all_bar();
      const int t_ = iv[2];
      if (t_ < 0) return false;
      r = t_ / d.nkpt;
      k = t_ - r * d.nkpt;
      const Point diff = minus(d, corner_of(d, r), point_of(d, k));
      for (int i = tid; i < rs; i += kThreads) {
        const int b = block_of(d, g, k, diff, i);
        slot[i] = b;
        if (b >= 0) iv[5] = taken;
      }
      all_bar();
    } while (iv[5] != taken);
    kc = umma::uniform(d.tc_kcount[r]);
    // ---- tile setup: blocks per slot, K keys, sphere keys of k, rows
    for (int i = tid; i < g.nwords; i += kThreads) bits[i] = 0u;
    for (int i = tid; i < iv[4]; i += kThreads) box[pkey[i]] = make_uint2(0u, 0u);   // the previous tile's points
    for (int i = tid; i < g.nkc * kTKC; i += kThreads) {
      int key = g.box_c;                         // padding: G2 = 0 (the B images are zero there)
      if (i < kc) {
        const char4 g2 = d.tc_klist[(size_t)r * d.tc_kpad + i];
        key += ((int)g2.x * g.by + (int)g2.y) * g.bz + (int)g2.z;
      }
      kkey[i] = key * 8;
    }
    for (int i = tid; i < rs; i += kThreads) {   // per slot of the region; x = -1: no block of this range
      const int b = slot[i];
      if (b < 0) {
        binfo[i] = make_int4(-1, 0, 0, 0);
        for (int n = 0; n < nb; ++n) binv[i * nb + n] = 0.f;
        continue;
      }
      const int4 blk = d.blocks[b];
      const long long qb = d.qblk_off[blk.z], nbq = d.qblk_off[blk.z + 1] - qb;
      const long long base = d.qvec_off[blk.z] - g.vbase;
      binfo[i] = make_int4(blk.z, blk.y, blk.w, 0);
      bptr[2 * i] = out + (size_t)(base + (b - qb) * nv * nv) * d.ng_max;
      bptr[2 * i + 1] = out + (size_t)(base + nbq * nv * nv + (b - qb) * nc * nc) * d.ng_max;
      for (int n = 0; n < nb; ++n) binv[i * nb + n] = scale[(size_t)d.nkpt * nb + (size_t)blk.y * nb + n];
    }
    all_bar();
    for (int i = warp; i < rs; i += kThreads / 32) {   // the union of the blocks' spheres, one warp per block
      const int b = slot[i];
      if (b < 0) continue;
      const int4 blk = d.blocks[b];
      const int gx = (blk.w & 3) - 1, gy = ((blk.w >> 2) & 3) - 1, gz = ((blk.w >> 4) & 3) - 1;
      const int ng = d.ngq[blk.z];
      const char4* gq = d.gq + (size_t)blk.z * d.ng_max;
      for (int p0_ = 0; p0_ < ng; p0_ += 128) {   // four loads in flight
        char4 gp[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) gp[u] = gq[min(p0_ + 32 * u + lane, ng - 1)];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int z = gp[u].z - gz + p2;
          atomicOr(&bits[((gp[u].x - gx + p0) * rb1 + gp[u].y - gy + p1) * g.wpl + (z >> 5)], 1u << (z & 31));
        }
      }
    }
    all_bar();
    n1 = d.npw[k];
    for (int i = tid; i < n1; i += kThreads) {
      const char4 gg = d.gk[(size_t)k * d.npw_max + i];
      pkey[i] = g.box_c + ((int)gg.x * g.by + (int)gg.y) * g.bz + (int)gg.z;
    }
    if (tid == 0) iv[4] = n1;
    if (warp == 0) {                             // rows in lexicographic order: neighbours in a warp gather neighbours
      int n = 0;
      for (int w0 = 0; w0 < g.nwords; w0 += 32) {
        const int w = w0 + lane;
        unsigned m = w < g.nwords ? bits[w] : 0u;
        const int cnt = __popc(m);
        int incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int t = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += t;
        }
        int pos = n + incl - cnt;
        const int line = w / g.wpl, x = line / rb1 - p0, y = line % rb1 - p1, z0 = (w % g.wpl) * 32 - p2;
        while (m) {
          rows[pos++] = make_char4((signed char)x, (signed char)y, (signed char)(z0 + __ffs(m) - 1), 0);
          m &= m - 1u;
        }
        n += __shfl_sync(0xffffffffu, incl, 31);
      }
      if (lane == 0) iv[3] = n;
    }
    all_bar();
    MT = umma::uniform(iv[3]);
    if (MT <= g.cap) {                           // (a larger union: per pass, below)
      for (int i0 = tid; i0 < MT * rs; i0 += 4 * kThreads) {   // four lookups in flight
        short v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int i = min(i0 + u * kThreads, MT * rs - 1), row = i / rs;
          v[u] = position(rows[row], binfo[i - row * rs]);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (i0 + u * kThreads < MT * rs) ptab[i0 + u * kThreads] = v[u];
      }
      all_bar();
    }
    nmt = (MT + 127) / 128;
    nch = (kc + kChunk - 1) / kChunk;
    return true;
  };

  if (role == 2) {                               // ---- gather: A tiles into tensor memory
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegGather));
    int sa = 0;                                  // A slot and its phase
    uint32_t aph = 0u;
    bool ok = true;
    while (next_tile()) {
      const int gt = tid - kG0 * 32, q4 = warp & 3;
      const uint32_t box_u = smem_u32(box);
      uint2 x[16];
      auto load16 = [&](uint32_t at_, int k0) {  // 16 K values of this row
        const int4* kp = reinterpret_cast<const int4*>(kkey + k0);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int4 t = kp[q];
          x[4 * q] = lds64(at_ + (uint32_t)t.x);
          x[4 * q + 1] = lds64(at_ + (uint32_t)t.y);
          x[4 * q + 2] = lds64(at_ + (uint32_t)t.z);
          x[4 * q + 3] = lds64(at_ + (uint32_t)t.w);
        }
      };
      auto pack16 = [&](uint32_t (&v)[32]) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          v[j] = __byte_perm(x[2 * j].x, x[2 * j + 1].x, 0x5410);        // Re hi
          v[8 + j] = __byte_perm(x[2 * j].y, x[2 * j + 1].y, 0x5410);    // Im hi
          v[16 + j] = __byte_perm(x[2 * j].x, x[2 * j + 1].x, 0x7632);   // Re lo
          v[24 + j] = __byte_perm(x[2 * j].y, x[2 * j + 1].y, 0x7632);   // Im lo
        }
      };
      for (int n = 0; n < nb; ++n) {             // valence bands, then conduction bands
        gather_bar();                            // every gather warp is done with the previous band
        {
          const float2* cn = coef + ((size_t)k * nb + n) * d.npw_max;
          const float a = scale[(size_t)k * nb + n];
          for (int i = gt; i < n1; i += kGThreads) {
            const float2 c = cn[i];
            box[pkey[i]] = make_uint2(split_word(c.x * a), split_word(-c.y * a));    // conj
          }
        }
        gather_bar();
        if (umma::uniform(*fail != 0)) ok = false;
        for (int mt = 0; mt < nmt; ++mt) {
          const int row = mt * 128 + q4 * 32 + lane;
          uint32_t at = box_u;                   // rows past the last one gather something and are dropped
          if (row < MT) {
            const char4 G = rows[row];
            at -= (uint32_t)((((int)G.x * g.by + (int)G.y) * g.bz + (int)G.z) * 8);
          }
          // the lookups of the next 16 K values are in flight while the last ones are packed and stored
          load16(at, 0);
          for (int c = 0; c < nch; ++c) {
            if (ok) {
              ok = umma::uniform(mbar_wait(smem_u32(empty_a + sa), aph ^ 1u));
              if (!ok) fail_now(fail, status);
            }
            if (ok) {
              asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
              const uint32_t ta = tmem + ((uint32_t)(q4 * 32) << 16) + a_col0 + (uint32_t)(sa * kACols_);
              const int k0 = c * kChunk, kn = min(c + 1, nch - 1) * kChunk;
              const bool two = SUB > 1 && kc - k0 > kTKC;
              uint32_t v[32];
              pack16(v);
              load16(at, k0 + 16);
              umma::tmem_st32(ta, v);
              pack16(v);
              load16(at, two ? k0 + kTKC : kn);
              umma::tmem_st32(ta + 32u, v);
              if (two) {
                pack16(v);
                load16(at, k0 + kTKC + 16);
                umma::tmem_st32(ta + 64u, v);
                pack16(v);
                load16(at, kn);
                umma::tmem_st32(ta + 96u, v);
              }
              asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
              asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
              __syncwarp();
              if (lane == 0) mbar_arrive(smem_u32(full_a + sa));
            }
            if (++sa == kAStages) {
              sa = 0;
              aph ^= 1u;
            }
          }
        }
      }
    }
  } else if (role == 3) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegIssue));
    unsigned copied = 0;                         // B producer: stages whose copies have been issued
    int st = 0, sa = 0;                          // B stage, A slot and accumulator, and their phases
    uint32_t bph = 0u, aph = 0u, cph = 0u, buf = 0u;
    bool ok = true;
    const bool leader = umma::elect_one();       // one lane for every MMA and commit of the warp: a commit tracks its own thread
    while (next_tile()) {
    if (warp == kB0) {                           // ---- B producer: the region's panel, two bulk copies per stage
      if (lane == 0) {
        for (int set = 0; set < 2; ++set) {
          const int nset = set ? nc : nv;
          const uint32_t half_bytes = (uint32_t)(rs * nset) * umma::kRow;
          for (int pass = 0; pass < nset * nmt; ++pass)
            for (int c = 0; c < nch; ++c) {
              if (ok && !mbar_wait(smem_u32(empty_b + st), bph ^ 1u)) {
                fail_now(fail, status);
                ok = false;
              }
              if (!ok) continue;
              const int np = min(SUB, (kc - c * kChunk + kTKC - 1) / kTKC);
              umma::mbar_arrive_expect_tx(smem_u32(full_b + st), 2 * np * half_bytes);
              for (int u = 0; u < np; ++u) {
                const uint32_t bh = smem_u32(sm + (size_t)st * g.stage_bytes + (size_t)u * g.sub_bytes);
                const unsigned char* p = bimg + panel_off(d, r, set, c * SUB + u, g.nkc);
                umma::bulk_g2s(bh, p, half_bytes, smem_u32(full_b + st));
                umma::bulk_g2s(bh + (uint32_t)(g.nmax * umma::kRow), p + half_bytes, half_bytes, smem_u32(full_b + st));
              }
              ++copied;
              if (++st == g.stages) {
                st = 0;
                bph ^= 1u;
              }
            }
        }
      }
      __syncwarp();
    } else if (warp < kB0) {                     // ---- MMA issue: the whole warp runs the loop, one lane issues
      // Two warps, one per accumulator (even and odd stages): a stage's three waits take ~300 cycles even when
      // everything is there, and run while the other warp's MMAs do.  Lanes 0-2 wait on one barrier each; the warp barrier
      // after the vote orders what they acquired before the MMAs of the issuing lane (a vote orders no memory).
      const uint32_t own = (uint32_t)(warp - kMmaWarp);
      unsigned p = pc;
      if (umma::uniform(*fail != 0)) ok = false;
      const uint64_t dstage0 = umma::smem_desc(umma::uniform(smem_u32(sm)));   // B stage st: + st stage_bytes / 16
      const uint32_t blo = (uint32_t)((g.nmax * umma::kRow) >> 4), bsub = (uint32_t)(g.sub_bytes >> 4);
      for (int set = 0; set < 2; ++set) {
        const int nset = set ? nc : nv;
        const uint32_t idesc = tcf::idesc_f16((rs * nset + 15) & ~15);
        for (int pass = 0; pass < nset * nmt; ++pass, ++p) {
          uint64_t* tf = tfull + 2 * (p & 1u);
          for (int c = 0; c < nch; ++c) {
            if (ok && buf == own) {
              const uint32_t bar = lane == 0 ? smem_u32(full_a + sa) : lane == 1 ? smem_u32(full_b + st)
                                                                                   : smem_u32(tempty + buf);
              ok = __all_sync(0xffffffffu, mbar_wait(bar, lane == 0 ? aph : lane == 1 ? bph : cph ^ 1u)) != 0;
              if (!ok && leader) fail_now(fail, status);
              __syncwarp();
            }
            if (!ok) continue;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint64_t db = dstage0 + (uint64_t)((st * g.stage_bytes) >> 4);
            const uint32_t a = tmem + a_col0 + (uint32_t)(sa * kACols_), d_re = tmem + own * kAcc;
            if (leader && buf == own) {
              const int left = kc - c * kChunk;
              if (SUB > 1 && left > 48)
                tcf::chunk_mmas_ts<2 * SUB>(d_re, d_re + kNCols, a, db, blo, bsub, idesc);
              else if (SUB > 1 && left > 32)
                tcf::chunk_mmas_ts<2 * SUB - 1>(d_re, d_re + kNCols, a, db, blo, bsub, idesc);
              else if (left > 16)
                tcf::chunk_mmas_ts<2>(d_re, d_re + kNCols, a, db, blo, bsub, idesc);
              else
                tcf::chunk_mmas_ts<1>(d_re, d_re + kNCols, a, db, blo, bsub, idesc);
              mma_commit(smem_u32(empty_a + sa));
              mma_commit(smem_u32(empty_b + st));
              mma_commit(smem_u32(tf + own));
            }
            __syncwarp();
            if (++sa == kAStages) {
              sa = 0;
              aph ^= 1u;
            }
            if (++st == g.stages) {
              st = 0;
              bph ^= 1u;
            }
            cph ^= buf;
            buf ^= 1u;
          }
        }
      }
    }
    }
    if (warp == kB0 && lane == 0 && *fail)       // copies still in flight after a failure
      for (unsigned c = copied > (unsigned)g.stages ? copied - g.stages : 0u; c < copied; ++c)
        if (!mbar_wait(smem_u32(full_b + c % (unsigned)g.stages), (c / g.stages) & 1u)) break;
    if (warp < kB0 && leader) {                  // tracks every MMA that this thread issued above
      mma_commit(smem_u32(drain + warp - kMmaWarp));
      if (!mbar_wait(smem_u32(drain + warp - kMmaWarp), 0u)) fail_now(fail, status);
    }
    __syncwarp();
  } else {                                       // ---- epilogue group: promote its passes, then write them
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegEpi));
    unsigned mine0 = 0u, mine1 = 0u;             // chunks this group has promoted from each accumulator
    while (next_tile()) {
      unsigned s = sc, p = pc;
      const int q4 = warp & 3;
      const uint32_t lane_addr = tmem + ((uint32_t)(q4 * 32) << 16);
      bool ok = true;
      for (int n = 0; n < nb; ++n) {
        const int set = n < nv ? 0 : 1, nset = set ? nc : nv, nn = set ? n - nv : n;
        const int ncols = rs * nset;
        for (int mt = 0; mt < nmt; ++mt, ++p) {
          if ((int)(p & 1u) != role) {
            s += (unsigned)nch;
            continue;
          }
          const int row = mt * 128 + q4 * 32 + lane;
          const bool valid = row < MT;
          short* pt = ptab + (size_t)(MT <= g.cap ? row : role * 128 + q4 * 32 + lane) * rs;
          if (MT > g.cap && valid) {
            const char4 G = rows[row];
#pragma unroll 4
            for (int b = 0; b < rs; ++b) pt[b] = position(G, binfo[b]);
          }
          float re[kNCols], im[kNCols];
#pragma unroll
          for (int j = 0; j < kNCols; ++j) re[j] = im[j] = 0.f;
          for (int c = 0; c < nch; ++c, ++s) {
            const int buf = (int)(s & 1u);
            if (ok) {
              ok = mbar_wait(smem_u32(tfull + 2 * role + buf), (buf ? mine1 : mine0) & 1u);
              if (!ok) fail_now(fail, status);
              ok = umma::uniform(ok);
            }
            mine0 += buf ? 0u : 1u;
            mine1 += buf ? 1u : 0u;
            if (!ok) continue;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t base = lane_addr + (uint32_t)(buf * kAcc);
#pragma unroll
            for (int j0 = 0; j0 < kNCols; j0 += 16) {
              if (j0 >= ncols) break;
              uint32_t v[16], u[16];
              umma::tmem_ld16(base + (uint32_t)j0, v);
              umma::tmem_ld16(base + (uint32_t)(kNCols + j0), u);
              asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
              for (int j = 0; j < 16; ++j) {
                re[j0 + j] += __uint_as_float(v[j]);
                im[j0 + j] += __uint_as_float(u[j]);
              }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(tempty + buf));
          }
          if (!ok || !valid) continue;
          const float ia = scale[(size_t)d.nkpt * nb + (size_t)k * nb + n];
          const float* ib = binv + (set ? nv : 0);
          const size_t first = (size_t)nn * nset * d.ng_max;
          auto write = [&](auto small) {
            constexpr bool S = decltype(small)::value;
            switch (nset) {
              case 1: write_pass<1, S>(re, im, ia, ib, bptr + set, pt, rs, nb, first, d.ng_max); break;
              case 2: write_pass<2, S>(re, im, ia, ib, bptr + set, pt, rs, nb, first, d.ng_max); break;
              case 3: write_pass<3, S>(re, im, ia, ib, bptr + set, pt, rs, nb, first, d.ng_max); break;
              default: write_pass<4, S>(re, im, ia, ib, bptr + set, pt, rs, nb, first, d.ng_max); break;
            }
          };
          if (ia < 1.f)
            write(std::true_type{});
          else
            write(std::false_type{});
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    __syncwarp();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
}

// ---------------------------------------------------------------- FP64 G = 0 overlaps of the diagonal blocks
// rho_nm^{kk}(0) = sum_G1 conj(c_nk(G1)) c_mk(G1), one warp per band product; q = 0 must be in the range.
__global__ void tcpair_diag_kernel(DevSys d, const float2* __restrict__ coef, float2* __restrict__ out,
                                   long long vbase) {
  const int k = blockIdx.x;
  const int b = d.blkidx[k];                     // q = 0 row of the table: the block (k, k)
  if (b < 0) return;
  const long long qb = d.qblk_off[0], nbq = d.qblk_off[1] - qb;
  const long long base = d.qvec_off[0] - vbase;
  const int nv = d.nv, nc = d.nc, n1 = d.npw[k];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int t = w; t < nv * nv + nc * nc; t += nw) {
    int a, bb;
    long long vec;
    if (t < nv * nv) {
      a = t / nv;
      bb = t % nv;
      vec = base + (b - qb) * nv * nv + t;
    } else {
      const int u = t - nv * nv;
      a = nv + u / nc;
      bb = nv + u % nc;
      vec = base + nbq * nv * nv + (b - qb) * nc * nc + u;
    }
    const float2* x = coef + ((size_t)k * d.nb + a) * d.npw_max;
    const float2* y = coef + ((size_t)k * d.nb + bb) * d.npw_max;
    double sr = 0.0, si = 0.0;
    for (int i = lane; i < n1; i += 32) {
      const float2 xv = x[i], yv = y[i];
      sr += (double)xv.x * yv.x + (double)xv.y * yv.y;      // conj(x) y
      si += (double)xv.x * yv.y - (double)xv.y * yv.x;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      sr += __shfl_xor_sync(0xffffffffu, sr, o);
      si += __shfl_xor_sync(0xffffffffu, si, o);
    }
    if (lane == 0) out[(size_t)vec * d.ng_max] = make_float2((float)sr, (float)si);
  }
}

// Panels per stage, ring depth and position-table rows.  Two panels (64 complex K per promotion and per hand-over of a
// stage) where two such stages and the table of the two groups' passes (256 rows) fit; one panel otherwise.  Two against
// one, ms (with the tiles from a counter): 27x27 sheet 1.03 / 1.13, 32x32 sheet 1.41 / 1.51, 5x5x5 4v4c 1.87 / 2.00, 12x12x12 144 q 45.3 / 47.9, 8x8x8 3v4c
// 9.9 / 10.6.  The table holds one and a half spheres of rows (512 to 1024) if it can: the rows are the union of
// spheres whose centres lie within a region of each other, and a larger union is looked up pass by pass.  The depth is
// even, so that a stage's slot always belongs to the same issue warp (which then sees every phase of the slot's
// barriers).  Depth 0: does not fit shared memory.
TpGeo tp_fit(const DevSys& d) {
  int cap0 = (d.ng_max * 3 / 2 + 127) / 128 * 128;
  cap0 = cap0 < 512 ? 512 : cap0 > 1024 ? 1024 : cap0;
  for (int sub = 2; sub >= 1; --sub)
    for (int cap = cap0; cap >= 256; cap -= 128)
      for (int st = sub == 2 ? 4 : kMaxStages; st >= (sub == 2 ? 2 : 4); st -= 2) {
        const TpGeo g = tp_geo(d, sub, st, cap);
        if (g.smem <= 227 * 1024) return g;
      }
  TpGeo g = tp_geo(d, 1, 2, 256);
  if (g.smem > 227 * 1024) g.stages = 0;
  return g;
}

struct TpWs {
  size_t bimg, scale, total;
};

TpWs tp_ws(const DevSys& d) {
  TpWs w;
  size_t o = 0;
  w.bimg = o; o += ((size_t)d.nkpt * d.nb * (d.tc_kpad / kTKC) * kImgRow + 255) & ~(size_t)255;
  w.scale = o; o += ((size_t)2 * d.nkpt * d.nb * sizeof(float) + 255) & ~(size_t)255;
  w.total = o;
  return w;
}

}  // namespace

// The tensor-core route needs a region of at most one N tile of columns and its tiles in shared memory.
int tcpair_valid(const DevSys& d) {
  if (d.nv > 4 || d.nc > 4) return 0;            // write_pass
  if ((long long)d.nkpt * d.tc_nreg >= 1ll << 31) return 0;   // deal_tiles
  if (d.tc_kpad < kTKC || d.tc_rsize < 1 || d.tc_rsize * (d.nv > d.nc ? d.nv : d.nc) > kNCols) return 0;
  return tp_fit(d).stages > 0 ? 1 : 0;
}

// Whether the direct set of [q_begin, q_end) goes to this kernel when the caller has not chosen one.  A tile is a k and
// a region of k'; it costs the same however few of the region's points have a block in the range, so the
// route needs tiles for every SM and columns in use: at least 304 tiles, and at least 30 of the 2 x 64 columns of a
// tile's two band sets on average (regions of the mesh k + q touches are counted at one k off the region grid).
// Measured, this kernel against gcorr_kernel (ms a call; the systems below the line pack in the call): 27x27 sheet 2v3c, 64 q
// (32 columns) 0.96 / 1.52; 32x32 sheet 3v3c, 64 q 1.31 / 2.62; 5x5x5 4v4c (40) 3.98 / 12.9 at 12 Ha and 0.33 / 0.30 at 3 Ha
// (62 points: a tile is mostly set-up); 8x8x8 3v4c (112) 9.7 / 50.1; below the line 4x4x4 3v3c (256 tiles) 0.146 /
// 0.117, 3x3x3 1v2c (27 tiles) 0.060 / 0.035, 7x7x7 2v2c, 49 q (28) 0.26 / 0.25 at 4 Ha (0.89 / 1.93 at 8.6 Ha: the line is
// drawn by columns alone).  With k-point symmetry only scattered representative blocks are left and the tiles are
// nearly empty.
int tcpair_preferred(const DevSys& d, int q_begin, int q_end) {
  if (!tcpair_valid(d) || d.nfill > 0) return 0;
  const int nqc = q_end - q_begin;
  int touched = d.tc_nreg;
  if (nqc < d.nq && d.tc_nreg <= 4096) {
    unsigned long long seen[64] = {};
    touched = 0;
    for (int q = q_begin; q < q_end; ++q) {
      const int i0 = (q / (d.nk2 * d.nk3) + d.tc_rg[0] / 2) % d.nk1, i1 = ((q / d.nk3) % d.nk2 + d.tc_rg[1] / 2) % d.nk2,
                i2 = (q % d.nk3 + d.tc_rg[2] / 2) % d.nk3;
      const int r = ((i0 / d.tc_rg[0]) * d.tc_nr[1] + i1 / d.tc_rg[1]) * d.tc_nr[2] + i2 / d.tc_rg[2];
      touched += (seen[r >> 6] >> (r & 63) & 1ull) ? 0 : 1;
      seen[r >> 6] |= 1ull << (r & 63);
    }
  }
  return (long long)d.nkpt * touched >= 304 && (long long)nqc * d.nb >= 30ll * touched ? 1 : 0;
}

size_t tcpair_ws_bytes(const DevSys& d) { return tcpair_valid(d) ? kWsSlack + tp_ws(d).total : 0; }

// Systems whose panels the real-space stage packs: those whose default route over the whole mesh is this kernel (where it
// is that of a part of the mesh it is that of the whole: the regions are of one size).  In the others a call with
// BSE_PD_TENSOR packs for itself.
int tcpair_packed(const DevSys& d) { return tcpair_preferred(d, 0, d.nq); }

// The tensor-route area ws (tcpair_ws_bytes) from coef (nkpt x nb x npw_max), and a copy of coef unless copy is NULL.
int launch_tcpair_pack(const DevSys& d, const void* coef, void* copy, void* ws, void* stream) {
  const TpWs w = tp_ws(d);
  unsigned char* base = ws_base(ws);
  tcpair_pack_kernel<<<(unsigned)(((long long)d.nkpt * d.nb + 7) / 8), 256, 0, (cudaStream_t)stream>>>(
      d, (const float2*)coef, (float2*)copy, (float*)(base + w.scale), base + w.bimg, d.tc_kpad / kTKC);
  return (int)cudaGetLastError();
}

// coef: the coefficient copy of the pair workspace; ws: the tensor-route area, packed by launch_tcpair_pack.  Both are
// only read.
int launch_tcpair(const DevSys& d, const void* coef, const void* ws, void* rho_dir, int q_begin, int q_end,
                  long long vbase, int* status, void* stream) {
  if (!tcpair_valid(d)) return (int)cudaErrorInvalidValue;
  TpGeo g = tp_fit(d);
  auto kernel = g.sub == 2 ? tcpair_kernel<2> : tcpair_kernel<1>;
  int dev = 0, num_sms = 0;
  int e = (int)cudaGetDevice(&dev);
  if (e) return e;
  if ((e = (int)cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, dev))) return e;
  if ((e = (int)cudaFuncSetAttribute((const void*)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024)))
    return e;
  cudaStream_t st = (cudaStream_t)stream;
  const TpWs w = tp_ws(d);
  const unsigned char* base = ws_base(const_cast<void*>(ws));
  g.q_begin = q_begin;
  g.nqc = q_end - q_begin;
  g.vbase = vbase;
  // a CTA lists kMine kThreads tiles a launch; an upper bound of the tiles with a block says how many launches
  long long diffs = std::min<long long>(d.nkpt, (long long)g.nqc * d.tc_rsize);
  g.table = (kList + kDealSums + diffs) * 4 <= (long long)g.stages * g.stage_bytes && d.nk1 <= 1024 && d.nk2 <= 1024 &&
            d.nk3 <= 1024;
  if (!g.table) diffs = d.nkpt;
  long long upto = 0;                            // tiles whose region reaches to k or beyond
  for (int r = 0; r < d.tc_nreg; ++r) {
    const int x = r / (d.tc_nr[1] * d.tc_nr[2]), y = (r / d.tc_nr[2]) % d.tc_nr[1], z = r % d.tc_nr[2];
    upto += (((x + 1) * d.tc_rg[0] - 1) * d.nk2 + (y + 1) * d.tc_rg[1] - 1) * (long long)d.nk3 + (z + 1) * d.tc_rg[2];
  }
  const long long most = std::min(d.tc_nreg * diffs, upto);
  const int grid = (int)std::min<long long>(most, num_sms);
  const long long step = (long long)kList * grid;
  for (g.share = 0; g.share * step < most; ++g.share) {
    kernel<<<(unsigned)grid, kThreads, g.smem, st>>>(d, (const float2*)coef, (const float*)(base + w.scale),
                                                     base + w.bimg, (float2*)rho_dir, g, status);
    if ((e = (int)cudaGetLastError())) return e;
  }
  if (q_begin == 0) {
    tcpair_diag_kernel<<<d.nkpt, 256, 0, st>>>(d, (const float2*)coef, (float2*)rho_dir, vbase);
    e = (int)cudaGetLastError();
  }
  return e;
}

}  // namespace bse
