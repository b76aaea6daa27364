// Fused torus passes of the FP32 / tensor-core plans: the odd-length DFTs along theta and phi
// (eqns dft_spatial / idft_spatial, Sec. 3.4.1) with the extension, phase, weight convolution and
// transposition steps, as matrix products on the tcgen05 tensor cores.
//
// Products.  All nodes are x_j = pi (2j+1)/N, N = 2L-1, and x_{N-1-j} = 2 pi - x_j, so folding the
// data about pi leaves real L x L matrices of cos(k x_j) and sin(k x_j) (Sec. 3.2's parity in
// theta; in phi the sums and differences of orders +-m or of mirrored samples):
//   theta inverse  column m of parity (-1)^{m+s}:  even  x(t) = F_0 + sum_{k>0} 2 cos(k x_t) F_k,
//                  odd  x(t) = i sum_{k>0} 2 sin(k x_t) F_k     (F_{m,-k} = (-1)^{m+s} F_{mk});
//   phi inverse    E(p) = sum_m cos(m x_p) (x_m + x_{-m}), O(p) = sum_m sin(m x_p) (x_m - x_{-m}),
//                  f(p) = E + i O, f(N-1-p) = E - i O;
//   phi forward    P_m = sum_p cos(m x_p) (f(p) + f(N-1-p)), Q_m = sum_p sin(m x_p) (f(p) - f(N-1-p)),
//                  X_{+-m} = P_m -+ i Q_m;
//   theta forward  H = W X with the real L x L matrix W of the extension, the DFT, the sin(theta) weight
//                  convolution and the fold of m' < 0 together (one matrix a parity; the odd one
//                  carries -i), applied to P and Q, which have the same parity as X_{+-m};
//   theta adjoint  the same with the transposed theta-inverse matrices.
// A pass is 8 B L^3 flops (24 B L^3 as split products), against two to four FFTs of 4L .. 8L points a row
// for the odd length (Bluestein's algorithm in shared memory, the passes this replaces).  GB300, alone, the
// four passes of an inverse and a forward (theta, phi, phi, theta), products against FFTs: L = 1024, B = 64
// 1.13, 1.18, 1.18, 1.17 ms against 2.08, 1.27, 1.64, 2.88; L = 2048, B = 16: inverse + forward 40.6 -> 33.4 ms as
// a whole.  Small band-limits, which would fill little of the tiles, take torus_small.cu (small_wanted).
//
// Precision.  Both operands are split x = hi + lo into two FP16 values (22 to 24 significant bits,
// the parts of an 11-bit significand each, as in a 3xTF32 split, at twice its rate) and the product
// is hi hi + hi lo + lo hi.  FP16's range is met by powers of two: a matrix carries one, the data
// one for every block of 16 rows and 64 K, taken from its largest magnitude (2^14 .. 2^15 after
// scaling; an element is off by at most 2^-24 of itself or 2^-39 of that largest one, which is in the
// same field and within 16 rings or 32 orders).  Each 32 K accumulate in a fresh tensor-memory
// segment, small products first, because the tensor core's FP32 accumulation truncates; the epilogue
// multiplies the segment by the block's power of two and adds it to running sums in registers (FMA,
// round to nearest).  Segments of 64 K would save the epilogue half of its reads but leave a larger
// error than the FFT passes had (round trip at L = 1024: 7.0e-7, against 6.5e-7 with the FFTs and
// 5.4e-7 with 32 K; 2-norms, from FP64).
//
// Layouts.  Data operands are K-major tiles of 128 rows x 32 K ("units", 16 KB): a row is 128
// bytes, 32 hi parts then 32 lo parts, in the 128-byte swizzle, moved by 1-D bulk copies.  A unit
// holds all chunks of its 128 rows back to back, and one FP32 scale for each block of 16 rows and 64 K.
//   theta inverse: units ((b, group of 64 |m| of one parity), part): rows eo * 64 + mi, K = m', of
//                  F_m + F_{-m} (eo = 0) and F_m - F_{-m} (1): the theta pass is linear and the same for m
//                  and -m, so that its outputs are the terms the phi pass wants;
//   phi inverse:   units ((b, 64 rings t), E or O): rows part * 64 + ti, K = |m|, even orders first;
//   phi forward:   units (even or odd, (b, 64 rings t)): rows part * 64 + ti, K = p;
//   theta forward: units ((b, group of 64 |m|), P or Q): rows part * 64 + mi, K = t.
// Each pass's epilogue writes the next pass's operand: a thread holds 64 consecutive K of a row, so
// a warp finds their scales, splits and stores them by itself.
#include "ssht_internal.h"
#include "bounds.cuh"
#include "tc_common.cuh"
#include "torus_matrices.cuh"

#include <algorithm>
#include <cmath>
#include <vector>

namespace ssht {
namespace {

using namespace tc;

constexpr int kUnitBytes = 128 * 128;  // one 32-K chunk of a unit, or a matrix tile
constexpr int kEpiWarps = 16;  // four a quarter of tensor memory's lanes, 64 columns each
// Five warpgroups: the producer and the MMA warp (and two idle ones), then the epilogue's.  640 threads
// are launched with 96 registers each; the first warpgroup gives some up so that the epilogue's 64
// running sums and a load of 16 columns stay in registers.
constexpr int kThreads = 128 + 32 * kEpiWarps;
constexpr int kRegsIssue = 48, kRegsEpilogue = 104;
static_assert(128 * kRegsIssue + 32 * kEpiWarps * kRegsEpilogue <= kThreads * 96, "register shares");
constexpr int kMaxStages = 6;
constexpr int kScaleSlots = 8;
static_assert(kScaleSlots >= kMaxStages + 2, "scale ring");
constexpr int kStageWarp = 4096;  // staging memory of an epilogue warp (passes that write operands)

enum Pass { kThetaInverse = 0, kPhiInverse = 1, kPhiForward = 2, kThetaForward = 3 };

// Sizes of a band-limit's operands.
struct Shape {
  int L, N;
  int nI;       // 128-row blocks of a matrix
  int nK;       // 32-K chunks in use, K = m', p or t
  int nKs;      // chunks stored: 64-K blocks
  int gE, gO;   // groups of 64 even and odd |m|
  int cE, cO;   // 32-K chunks in use of the even and the odd |m|
  int nT;       // groups of 64 rings
  __host__ __device__ int G() const { return gE + gO; }
  __host__ __device__ int nKm() const { return 2 * (gE + gO); }  // chunks stored, K = |m|
};

Shape make_shape(int L) {
  Shape s;
  s.L = L;
  s.N = 2 * L - 1;
  s.nI = (L + 127) / 128;
  s.nK = (L + 31) / 32;
  s.nKs = 2 * ((L + 63) / 64);
  const int nE = (L + 1) / 2, nO = L / 2;
  s.gE = (nE + 63) / 64;
  s.gO = (nO + 63) / 64;
  s.cE = (nE + 31) / 32;
  s.cO = (nO + 31) / 32;
  s.nT = (L + 63) / 64;
  return s;
}

// A data operand: its units of `chunks` 16 KB tiles and, behind them, the rows' scales.
struct Operand {
  uint8_t* x;
  float* scale;   // [unit][chunks / 2][8]
  long long units;
  int chunks;
};

size_t operand_bytes(long long units, int chunks) {
  return (size_t)units * chunks * kUnitBytes + (size_t)units * (chunks / 2) * 8 * sizeof(float);
}
Operand operand(void* base, long long units, int chunks) {
  Operand o;
  o.x = (uint8_t*)base;
  o.scale = (float*)((uint8_t*)base + (size_t)units * chunks * kUnitBytes);
  o.units = units;
  o.chunks = chunks;
  return o;
}

// Scales, splits and stores the 64 K values x[0..63] of 32 rows, one a lane (K block kb): each chunk's
// rows are put together in the warp's staging memory (4 KB, in the tile's layout) and leave by a
// bulk copy, which runs on beside the next tile.  (Stored by the threads themselves, 16
// bytes a lane 128 bytes apart, they took 17,000 clocks a tile of 128 x 256 outputs, half as much as
// its products at K = 1024.)  srow: the lane's row in the buffer, row: in the unit (the same modulo
// 8); LANES16: the lanes of a block of 16 rows are 16 in a row (or every other one); piece p of the buffer, bytes [p, p + 1) * 4096 / np, goes to tile row prow[p] of unit punit[p]
// (none if punit[p] < 0).
template <int NP, bool LANES16>
__device__ __forceinline__ void store_rows64(const Operand& o, uint8_t* stage, int lane, long long unit, int kb, int srow,
                                             int row, bool live, const long long (&punit)[NP], const int (&prow)[NP],
                                             const float* x) {
  float amax = 0.f;
#pragma unroll
  for (int k = 0; k < 64; ++k) amax = fmaxf(amax, fabsf(x[k]));
#pragma unroll
  for (int d = LANES16 ? 1 : 2; d < (LANES16 ? 16 : 32); d <<= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, d));
  float sc;
  const float up = block_power(amax, &sc);
  if (live && (row & 15) == 0 && in_bounds(unit, o.units, kbTorusTile) && in_bounds(kb, o.chunks / 2, kbTorusTile))
    o.scale[((size_t)unit * (o.chunks / 2) + kb) * 8 + (row >> 4)] = sc;
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    if (lane == 0) bulk_wait_read<0>();  // the copy that read the buffer last has done so
    __syncwarp();
    uint8_t* t = stage + srow * 128;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      uint4 h, l;
      const float* v = x + 32 * c + 8 * q;
      split2(v[0] * up, v[1] * up, &h.x, &l.x);
      split2(v[2] * up, v[3] * up, &h.y, &l.y);
      split2(v[4] * up, v[5] * up, &h.z, &l.z);
      split2(v[6] * up, v[7] * up, &h.w, &l.w);
      *(uint4*)(t + (((q ^ srow) & 7) << 4)) = h;
      *(uint4*)(t + ((((q + 4) ^ srow) & 7) << 4)) = l;
    }
    fence_proxy_async();
    __syncwarp();
    if (lane == 0) {
#pragma unroll
      for (int p = 0; p < NP; ++p)
        if (punit[p] >= 0 && in_bounds(punit[p], o.units, kbTorusTile) && in_bounds(kb, o.chunks / 2, kbTorusTile))
          bulk_s2g(o.x + ((size_t)punit[p] * o.chunks + 2 * kb + c) * kUnitBytes + prow[p] * 128,
                   stage + p * (4096 / NP), 4096 / NP);
      bulk_commit();
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Packing of the operands that no pass's epilogue writes: a CTA takes 16 rows (a warp each) and 128 K
// ---------------------------------------------------------------------------------------------

// A warp's lanes hold four terms (the real and imaginary parts of a sum and a difference, each a row of its
// own) of K = 2 lane and 2 lane + 1 in each of two 64-K blocks, v[block][term][2]; the CTA's 16 warps are the 16
// rows of the blocks that share a power of two.  The split parts are put together in shared memory in the
// tiles' layout and leave as 2 KB bulk copies, one a term and chunk (stored by the threads, 4 bytes a lane,
// the packing of L = 1024, B = 64 took 0.456 ms, now 0.397 by theta and 0.442 by phi; at L = 512, B = 32 60 us
// and 53 / 55 us; bound by HBM traffic and the conversions).  Term i goes to rows row0[i] .. row0[i] + 15 of unit[i].
__device__ __forceinline__ void pack_rows16(const Operand& o, const float (&v)[2][4][2], int kb0, const long long (&unit)[4],
                                            const int (&row0)[4], uint8_t* sm, float (*smax)[8]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t mx[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float m = fmaxf(fabsf(v[i >> 2][i & 3][0]), fabsf(v[i >> 2][i & 3][1]));
    mx[i] = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
  }
  if (lane == 0) {
#pragma unroll
    for (int i = 0; i < 8; ++i) smax[warp][i] = __uint_as_float(mx[i]);
  }
  __syncthreads();
  const uint32_t off = sw128(warp, 4 * (lane & 15));
  float mine = 0.f;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint32_t m = __reduce_max_sync(0xffffffffu, __float_as_uint(smax[lane & 15][i]));
    float sc;
    const float up = block_power(__uint_as_float(m), &sc);
    if (lane == i) mine = sc;
    uint32_t h, l;
    split2(up * v[i >> 2][i & 3][0], up * v[i >> 2][i & 3][1], &h, &l);
    // [term][block][chunk]: 16 rows of 128 bytes
    uint8_t* t = sm + (((i & 3) * 4 + 2 * (i >> 2) + (lane >> 4)) << 11);
    *(uint32_t*)(t + off) = h;
    *(uint32_t*)(t + (off ^ 64u)) = l;
  }
  const int nkb = o.chunks / 2;
  if (warp == 0 && lane < 8 && kb0 + (lane >> 2) < nkb) {
    const int i = lane & 3;
    if (in_bounds(unit[i], o.units, kbTorusTile))
      o.scale[((size_t)unit[i] * nkb + kb0 + (lane >> 2)) * 8 + (row0[i] >> 4)] = mine;
  }
  fence_proxy_async();
  __syncthreads();
  if (warp == 0) {
    if (lane < 16 && kb0 + ((lane >> 1) & 1) < nkb) {
      const int i = lane >> 2;
      if (in_bounds(unit[i], o.units, kbTorusTile))
        bulk_s2g(o.x + ((size_t)unit[i] * o.chunks + 2 * kb0 + (lane & 3)) * kUnitBytes + row0[i] * 128, sm + (lane << 11), 2048);
    }
    bulk_commit();
    bulk_wait_read<0>();
  }
}

// F half rows [b][m + Lp][m'] -> theta-inverse units F_m +- F_{-m} (m = 0: F_0 and 0); a CTA takes 16
// orders |m| of one parity.  blockIdx.x: (b, parity, 16 orders), blockIdx.y: 128 K.
__global__ void __launch_bounds__(512) pack_theta_kernel(Shape sh, int B, const float2* __restrict__ F, Operand o,
                                                         long long in_n) {
  __shared__ __align__(1024) uint8_t sm[16 * 2048];
  __shared__ float smax[16][8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, kb0 = 2 * blockIdx.y;
  const int nq = ((sh.L + 1) / 2 + 15) / 16, nqo = (sh.L / 2 + 15) / 16;  // blocks of even and of odd orders
  const int b = blockIdx.x / (nq + nqo), r = blockIdx.x - b * (nq + nqo), odd = r >= nq ? 1 : 0;
  const int q0 = 16 * (r - odd * nq), am = 2 * (q0 + warp) + odd;
  const long long rp = ((long long)b * sh.N + sh.L - 1 + am) * sh.L, rm = ((long long)b * sh.N + sh.L - 1 - am) * sh.L;
  float v[2][4][2];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int k = 64 * (kb0 + (i >> 1)) + 2 * lane + (i & 1);
    float2 x = make_float2(0.f, 0.f), y = x;
    if (am < sh.L && k < sh.L && in_bounds(rp + k, in_n, kbTorusIn)) x = __ldg(&F[rp + k]);
    if (am < sh.L && k < sh.L && am > 0 && in_bounds(rm + k, in_n, kbTorusIn)) y = __ldg(&F[rm + k]);
    v[i >> 1][0][i & 1] = x.x + y.x;
    v[i >> 1][1][i & 1] = x.y + y.y;
    v[i >> 1][2][i & 1] = am > 0 ? x.x - y.x : 0.f;
    v[i >> 1][3][i & 1] = am > 0 ? x.y - y.y : 0.f;
  }
  const long long unit = 2 * ((long long)b * sh.G() + (odd ? sh.gE : 0) + (q0 >> 6));
  const int row = q0 & 63;
  pack_rows16(o, v, kb0, {unit, unit + 1, unit, unit + 1}, {row, row, 64 + row, 64 + row}, sm, smax);
}

// Samples f [b][t][p] -> phi-forward units: sums and differences of mirrored samples (p = L - 1 is
// its own mirror image); a CTA takes 16 rings.  blockIdx.x: (b, 16 rings), blockIdx.y: 128 K.
__global__ void __launch_bounds__(512) pack_phi_kernel(Shape sh, int B, const float2* __restrict__ f, Operand o,
                                                       long long in_n) {
  __shared__ __align__(1024) uint8_t sm[16 * 2048];
  __shared__ float smax[16][8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, kb0 = 2 * blockIdx.y;
  const int nt = (sh.L + 15) / 16, b = blockIdx.x / nt, t0 = 16 * (blockIdx.x - b * nt), t = t0 + warp;
  const long long at = ((long long)b * sh.L + t) * sh.N;
  float v[2][4][2];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int p = 64 * (kb0 + (i >> 1)) + 2 * lane + (i & 1);
    float2 x = make_float2(0.f, 0.f), y = x;
    if (t < sh.L && p < sh.L && in_bounds(at + p, in_n, kbTorusIn)) x = __ldg(&f[at + p]);
    if (t < sh.L && p < sh.L - 1 && in_bounds(at + sh.N - 1 - p, in_n, kbTorusIn)) y = __ldg(&f[at + sh.N - 1 - p]);
    v[i >> 1][0][i & 1] = x.x + y.x;
    v[i >> 1][1][i & 1] = x.y + y.y;
    v[i >> 1][2][i & 1] = p < sh.L - 1 ? x.x - y.x : 0.f;
    v[i >> 1][3][i & 1] = p < sh.L - 1 ? x.y - y.y : 0.f;
  }
  const long long half = o.units / 2, unit = (long long)b * sh.nT + (t0 >> 6);
  const int row = t0 & 63;
  pack_rows16(o, v, kb0, {unit, unit, half + unit, half + unit}, {row, 64 + row, row, 64 + row}, sm, smax);
}

// ---------------------------------------------------------------------------------------------
// The product
// ---------------------------------------------------------------------------------------------
struct TgArgs {
  Shape sh;
  int s, B;               // B: fields of this slice
  int b0;                 // its first field (theta forward into tiles)
  int stages;
  int ntiles;             // work items: column tile * row_tiles + row tile
  int row_tiles;          // row blocks, or pairs of them
  const uint8_t* A[2];    // matrix of parity (or E / O, P / Q) 0 and 1: tiles [i][chunk stored]
  int a_chunks;           // chunks stored a row block
  float alpha;            // power of two undoing the matrix's scale (less the 2^-14 in the rows' scales)
  Operand in, out;        // out: the next pass's operand (theta inverse, phi forward)
  float2* f;              // phi inverse: samples; theta forward without tiles: H
  long long f_n;
  TileOut to;             // theta forward: the projection's data tiles (mode 0: H)
  int* status;
  long long wait_ns;
};

// What a work item multiplies.
struct Item {
  int i, j;           // row tile, column tile
  int a;              // matrix
  long long u0, u1;   // units of columns 0..127 and 128..255
};

template <int MODE>
__device__ __forceinline__ Item tile_item(const TgArgs& a, int w) {
  Item it;
  it.j = w / a.row_tiles;
  it.i = w - it.j * a.row_tiles;
  if constexpr (MODE == kThetaInverse || MODE == kThetaForward) {
    const int g = it.j % a.sh.G();
    it.a = ((g < a.sh.gE ? 0 : 1) + a.s) & 1;  // parity of m + s
    it.u0 = 2ll * it.j;
    it.u1 = it.u0 + 1;
  } else if constexpr (MODE == kPhiInverse) {
    it.a = 0;
    it.u0 = 2ll * it.j;
    it.u1 = it.u0 + 1;
  } else {
    // pairs of rings' units, of the sums first, then of the differences
    const int per = a.B * a.sh.nT, pairs = (per + 1) / 2;
    it.a = it.j < pairs ? 0 : 1;
    const int p = it.j - it.a * pairs;
    it.u0 = (long long)it.a * per + 2 * p;
    it.u1 = 2 * p + 1 < per ? it.u0 + 1 : it.u0;  // the last one may be alone: its second half is not used
  }
  return it;
}

// 64-K blocks of a pass and the chunks in use of block kb: one or two.
template <int MODE> __device__ __forceinline__ int k_blocks(const Shape& sh) {
  return MODE == kPhiInverse ? sh.G() : sh.nKs / 2;
}
template <int MODE> __device__ __forceinline__ int block_chunks(const Shape& sh, int kb) {
  const int left = MODE != kPhiInverse ? sh.nK - 2 * kb : kb < sh.gE ? sh.cE - 2 * kb : sh.cO - 2 * (kb - sh.gE);
  return left >= 2 ? 2 : 1;
}

// The 64 accumulator columns of epilogue warp group cg, as four groups g of 16: theta inverse and phi
// forward take half a unit each (64 K of the next operand's rows); phi inverse and theta forward take
// 16 rows of each half of both units, so that a thread has all four terms of its outputs.
template <int MODE>
__device__ __forceinline__ int group_col(int cg, int g) {
  if constexpr (MODE == kThetaInverse || MODE == kPhiForward) return 64 * cg + 16 * g;
  return 64 * g + 16 * cg;
}

// Theta forward's stores of the rows m' of a warp's lanes (one 32-K chunk of the projection) into the data
// tiles of 16 orders |m| = am0, am0 + 2, .. (acc: H_{+m} re, im, H_{-m} re, im, 16 each); the whole warp calls
// it.  The rows of m and -m share a power of two.  Orders past L - 1 are computed and not stored, so that
// the 16 orders' chains of reduction, split and stores overlap.
template <bool BF>
__device__ __forceinline__ void put_orders(const TileOut& to, int sl, int am0, int row, int lane, int L, int half, int r0,
                                           float sgn, const float* acc) {
  const int pbytes = to.NC * 128, orders = min(16, (L - am0 + 1) >> 1);
  const size_t tb = (size_t)kParts<BF> * pbytes;
  const long long slice_tiles = (long long)(to.xslice / tb), n = (long long)(to.xbytes / tb);
  const long long tix0 = sl * slice_tiles + (long long)am0 * to.nC + (row >> 5);
  const bool rows_ok = in_bounds(half + r0 + 1, to.NC, kbPutTile);
  float mine = 0.f;
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const long long tix = tix0 + 2 * k * to.nC;
    const float v[4] = {acc[k], acc[16 + k], sgn * acc[32 + k], sgn * acc[48 + k]};
    float sc = 0.f;
    const float up = BF ? 1.f : warp_power(fmaxf(fmaxf(fabsf(v[0]), fabsf(v[1])), fmaxf(fabsf(v[2]), fabsf(v[3]))), &sc);
    if (lane == k) mine = sc;
    uint8_t* tile = to.X + (size_t)tix * tb;
    const bool ok = k < orders && rows_ok && in_bounds(tix, n, kbPutTile);
    put_rows2<BF>(tile, pbytes, r0, lane, v[0], v[1], up, ok);
    put_rows2<BF>(tile, pbytes, half + r0, lane, v[2], v[3], up, ok);
  }
  const long long tix = tix0 + 2 * lane * to.nC;  // lane k: order k's scales
  const bool own = lane < orders && rows_ok && in_bounds(tix, n, kbPutTile);
  if (!BF && own) {
    float* sc = to.scale + (size_t)tix * half;
    sc[r0 >> 1] = mine;
    sc[(half + r0) >> 1] = mine;
  }
}

// Persistent, one CTA an SM; the row blocks of a column tile are consecutive items, so that its
// data is read from HBM about once and by the other row blocks from L2, where the matrices stay too
// (4 bytes an entry: 4 MB each at L = 1024).  A tile is 128 x 256 outputs a CTA.
//
// A 32-K chunk is 768 clocks of tensor work on 48 KB of operands (phi inverse: 64 KB).  PAIR: two CTAs
// of a cluster share each product (cta_group::2) of 256 rows, each holding its 128 rows of the matrix and
// one of the two units, which cuts the copies to 32 KB (48 KB) a chunk.  The leader issues the products;
// the other CTA's copies are reported to it by that CTA's second warp.  One CTA alone where there is one
// row block only.  What bounds it: the tensor pipe (80 - 85 % of the 768 clocks' rate at L = 1024, B = 64),
// then the tile's last step, whose conversion and stores the next tile's first two chunks overlap.
template <int MODE, bool PAIR>
__device__ __forceinline__ void torus_gemm(const TgArgs& a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  constexpr bool DUAL = MODE == kPhiInverse;
  constexpr int A_BYTES = (DUAL ? 2 : 1) * kUnitBytes;
  constexpr int X_BYTES = (PAIR ? 1 : 2) * kUnitBytes;  // PAIR: one unit, or half of each (DUAL)
  constexpr int STAGE = A_BYTES + X_BYTES;
  const int STAGES = a.stages;
  // full: this CTA's copies of a stage have landed; peer_full (leader): the other CTA's
  __shared__ __align__(8) uint64_t full[kMaxStages], peer_full[kMaxStages], empty[kMaxStages], seg_full[2], seg_empty[2],
      done_bar;
  // the scales of a 64-K block's 16 blocks of columns: a ring that the producer fills ahead of the
  // products.  Slot reuse needs no barrier: when the producer fills chunk n, chunk n - STAGES has been
  // multiplied, so the epilogue has released chunk n - STAGES - 2 and read the scales up to it, at most
  // kScaleSlots blocks back.
  __shared__ __align__(16) float scales[kScaleSlots][16];
  __shared__ __align__(8) uint64_t scale_full[kScaleSlots];
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = PAIR ? cluster_rank() : 0u;
  if (warp == 1) {
    if constexpr (PAIR) tmem_alloc_pair(&tmem_base, 512);
    else tmem_alloc(&tmem_base, 512);
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&peer_full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int k = 0; k < 2; ++k) {
      mbar_init(&seg_full[k], 1);
      mbar_init(&seg_empty[k], (PAIR ? 2 : 1) * kEpiWarps);
    }
    for (int k = 0; k < kScaleSlots; ++k) mbar_init(&scale_full[k], 1);
    mbar_init(&done_bar, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  if constexpr (PAIR) cluster_sync();
  fence_after();
  const uint32_t tbase = tmem_base;
  volatile int* abort = &abort_flag;
  const Shape& sh = a.sh;
  const int nkb = k_blocks<MODE>(sh), nchunk = MODE == kPhiInverse ? sh.cE + sh.cO : sh.nK;
  const int w0 = PAIR ? blockIdx.x >> 1 : blockIdx.x, wstep = PAIR ? gridDim.x >> 1 : gridDim.x;

  if (warp < 4) {
    regs_dec<kRegsIssue>();
    // The issuing warps run their loops as whole warps, one elected lane issuing: the addresses and
    // descriptors then stay in uniform registers (a single lane's loop took 70 clocks a product to issue).
    if (warp == 0) {
      // ---- producer ----
      const bool one = elect_one();
      int s = 0, ph = 1, is = 0, nscale = 0;  // stage, parity its empty barrier is waited for, segment
      uint32_t used = 0, uph = 0;  // stages that were filled, and the parity of their last fill
      for (int w = w0; w < a.ntiles && !*abort; w += wstep) {
        const Item itm = tile_item<MODE>(a, w);
        const bool ok_u = in_bounds(itm.u0, a.in.units, kbTorusTile) && in_bounds(itm.u1, a.in.units, kbTorusTile);
        const uint8_t* x0 = a.in.x + (size_t)(ok_u ? itm.u0 : 0) * a.in.chunks * kUnitBytes;
        const uint8_t* x1 = a.in.x + (size_t)(ok_u ? itm.u1 : 0) * a.in.chunks * kUnitBytes;
        // a pair's second row block may not exist: its products go unused
        const int ib = min(PAIR ? 2 * itm.i + (int)rank : itm.i, sh.nI - 1);
        const size_t arow = (size_t)ib * a.a_chunks * kUnitBytes;
        const uint8_t* m0 = a.A[DUAL ? 0 : itm.a] + arow;
        const uint8_t* m1 = a.A[1] + arow;
        const float* s0 = a.in.scale + (size_t)(ok_u ? itm.u0 : 0) * (a.in.chunks / 2) * 8;
        const float* s1 = a.in.scale + (size_t)(ok_u ? itm.u1 : 0) * (a.in.chunks / 2) * 8;
        bool ok = true;
        for (int kb = 0; kb < nkb && ok; ++kb, ++is) {
          const int nc = block_chunks<MODE>(sh, kb);
          for (int c = 2 * kb; c < 2 * kb + nc; ++c) {
            if (!__all_sync(0xffffffffu, mbar_wait(&empty[s], ph, abort, a.wait_ns))) {
              *abort = 1;
              ok = false;
              break;
            }
            if (c == 2 * kb) nscale = is + 1;
            if (one) {
              if (c == 2 * kb) {
                const int slot = is & (kScaleSlots - 1);
                mbar_expect_tx(&scale_full[slot], 64);
                bulk_g2s(scales[slot], s0 + kb * 8, 32, &scale_full[slot]);
                bulk_g2s(scales[slot] + 8, s1 + kb * 8, 32, &scale_full[slot]);
              }
              uint8_t* st = smem + s * STAGE;
              const size_t co = (size_t)c * kUnitBytes;
              mbar_expect_tx(&full[s], (uint32_t)STAGE);
              bulk_g2s(st, m0 + co, kUnitBytes, &full[s]);
              if constexpr (DUAL) bulk_g2s(st + kUnitBytes, m1 + co, kUnitBytes, &full[s]);
              if constexpr (!PAIR) {
                bulk_g2s(st + A_BYTES, x0 + co, kUnitBytes, &full[s]);
                bulk_g2s(st + A_BYTES + kUnitBytes, x1 + co, kUnitBytes, &full[s]);
              } else if constexpr (DUAL) {
                const size_t ho = rank * (kUnitBytes / 2);
                bulk_g2s(st + A_BYTES, x0 + co + ho, kUnitBytes / 2, &full[s]);
                bulk_g2s(st + A_BYTES + kUnitBytes / 2, x1 + co + ho, kUnitBytes / 2, &full[s]);
              } else {
                bulk_g2s(st + A_BYTES, (rank ? x1 : x0) + co, kUnitBytes, &full[s]);
              }
            }
            used |= 1u << s;
            uph = (uph & ~(1u << s)) | ((uint32_t)(ph ^ 1) << s);
            if (++s == STAGES) {
              s = 0;
              ph ^= 1;
            }
          }
        }
      }
      // drain: every issued copy must have landed before the CTA leaves
      for (int k = 0; k < STAGES; ++k)
        if ((used >> k) & 1u) mbar_wait(&full[k], (uph >> k) & 1u, nullptr, kDrainNs);
      for (int k = max(0, nscale - kScaleSlots); k < nscale; ++k)
        mbar_wait(&scale_full[k % kScaleSlots], (k / kScaleSlots) & 1, nullptr, kDrainNs);
    } else if (PAIR && rank == 1 && warp == 1) {
      // ---- the second CTA of a pair: tell the leader which stages have landed here ----
      const bool one = elect_one();
      const uint32_t pf = peer_addr(smem_u32(peer_full), 0);
      int s = 0, ph = 0;
      for (int w = w0; w < a.ntiles && !*abort; w += wstep) {
        for (int c = 0; c < nchunk; ++c) {
          if (!__all_sync(0xffffffffu, mbar_wait(&full[s], ph, abort, a.wait_ns))) {
            *abort = 1;
            break;
          }
          if (one) mbar_arrive_peer(pf + 8 * s);
          if (++s == STAGES) {
            s = 0;
            ph ^= 1;
          }
        }
      }
    } else if (warp == 1) {
      // ---- MMA issuer: one tensor-memory segment a chunk; parts hi at byte 0, lo at byte 64 of a
      // row, K = 16 (32 bytes) an instruction; the small products (hi lo, lo hi) first ----
      const uint32_t idesc = idesc_f16(PAIR ? 256 : 128, DUAL ? 128 : 256);
      const bool one = elect_one();
      const uint32_t lo0 = (smem_u32(smem) >> 4) + kDescLow;
      int s = 0, ph = 0, seg = 0, sph = 1;
      for (int w = w0; w < a.ntiles && !*abort; w += wstep) {
        for (int c = 0; c < nchunk; ++c) {
          const bool here = mbar_wait(&seg_empty[seg], sph, abort, a.wait_ns) && mbar_wait(&full[s], ph, abort, a.wait_ns) &&
                            (!PAIR || mbar_wait(&peer_full[s], ph, abort, a.wait_ns));
          if (!__all_sync(0xffffffffu, here)) {
            *abort = 1;
            break;
          }
          fence_after();
          if (one) {
            const uint32_t dt = tbase + (uint32_t)(seg * 256);
            const uint32_t la = lo0 + (uint32_t)(s * (STAGE >> 4)), lb = la + (A_BYTES >> 4);
#pragma unroll
            for (int q = 0; q < 3; ++q) {
              const uint32_t pa = q == 1 ? 4u : 0u, pb = q == 0 ? 4u : 0u;  // 64 bytes
#pragma unroll
              for (int kk = 0; kk < 2; ++kk) {
                const uint32_t acc = (q == 0 && kk == 0) ? 0u : 1u;
                mma_f16_lo<PAIR>(dt, la + pa + 2 * kk, lb + pb + 2 * kk, idesc, acc);
                if constexpr (DUAL)
                  mma_f16_lo<PAIR>(dt + 128, la + (kUnitBytes >> 4) + pa + 2 * kk, lb + (X_BYTES >> 5) + pb + 2 * kk, idesc, acc);
              }
            }
            if constexpr (PAIR) {
              mma_commit_pair(&empty[s]);
              mma_commit_pair(&seg_full[seg]);
            } else {
              mma_commit(&empty[s]);
              mma_commit(&seg_full[seg]);
            }
          }
          __syncwarp();
          if (++s == STAGES) {
            s = 0;
            ph ^= 1;
          }
          seg ^= 1;
          if (seg == 0) sph ^= 1;
        }
      }
      // every issued MMA has completed before the CTA (the pair) leaves
      if (one) {
        if constexpr (PAIR) mma_commit_pair(&done_bar);
        else mma_commit(&done_bar);
      }
      __syncwarp();
      mbar_wait(&done_bar, 0, nullptr, kDrainNs);
    }
  } else {
    // ---- epilogue ----
    regs_inc<kRegsEpilogue>();
    const int q = warp & 3;          // tensor-memory lane quarter this warp may access
    const int cg = (warp - 4) >> 2;  // its 64 columns
    const int L = sh.L;
    const uint32_t tq = tbase + ((uint32_t)(q * 32) << 16);
    const uint32_t leader_empty = PAIR ? peer_addr(smem_u32(seg_empty), 0) : 0u;
    uint8_t* stage = smem + STAGES * STAGE + (warp - 4) * kStageWarp;
    int is = 0, seg = 0, sph = 0;
    for (int w = w0; w < a.ntiles && !*abort; w += wstep) {
      const Item itm = tile_item<MODE>(a, w);
      // theta inverse, odd parity: the factor i makes the real part of -im and the imaginary one of re
      const float al = (MODE == kThetaInverse && itm.a && cg >= 2) ? -a.alpha : a.alpha;
      float acc[64];
#pragma unroll
      for (int k = 0; k < 64; ++k) acc[k] = 0.f;
      bool ok = true;
      for (int kb = 0; kb < nkb && ok; ++kb, ++is) {
        const int nc = block_chunks<MODE>(sh, kb), slot = is & (kScaleSlots - 1);
        float sc[4];
        for (int c = 0; c < nc; ++c) {
          if (c == 0) {
            ok = mbar_wait(&scale_full[slot], (is / kScaleSlots) & 1, abort, a.wait_ns);
#pragma unroll
            for (int g = 0; g < 4; ++g) sc[g] = scales[slot][group_col<MODE>(cg, g) >> 4];
          }
          if (!ok || !mbar_wait(&seg_full[seg], sph, abort, a.wait_ns)) {
            *abort = 1;
            ok = false;
            break;
          }
          fence_after();
          const uint32_t ts = tq + (uint32_t)(seg * 256);
#pragma unroll
          for (int g = 0; g < 4; g += 2) {
            uint32_t v[32];
            tmem_ld16_nowait(ts + group_col<MODE>(cg, g), v);
            tmem_ld16_nowait(ts + group_col<MODE>(cg, g + 1), v + 16);
            tmem_wait_ld();
            if (g == 2) {  // the segment is read: free it before the last sums
              fence_before();
              __syncwarp();
              if (lane == 0) {
                if constexpr (PAIR) mbar_arrive_peer(leader_empty + 8 * seg);
                else mbar_arrive(&seg_empty[seg]);
              }
            }
#pragma unroll
            for (int k = 0; k < 32; ++k)
              acc[16 * g + k] = fmaf(__uint_as_float(v[k]), sc[g + (k >> 4)], acc[16 * g + k]);
          }
          seg ^= 1;
          if (seg == 0) sph ^= 1;
        }
      }
      if (!ok) break;
#pragma unroll
      for (int k = 0; k < 64; ++k) acc[k] *= al;
      const int row0 = (PAIR ? 2 * itm.i + (int)rank : itm.i) * 128 + q * 32, row = row0 + lane;  // t, p, m or m'
      if (row0 >= 128 * sh.nI) continue;
      if constexpr (MODE == kThetaInverse) {
        // the terms eo = cg mod 2 of part cg / 2 of 64 orders of one parity
        if ((row0 >> 6) >= sh.nT) continue;  // the whole warp
        const int b = itm.j / sh.G(), g = itm.j - b * sh.G();
        const int cls = g < sh.gE ? 0 : 1, gi = cls ? g - sh.gE : g;
        const int left = ((cls ? L / 2 : (L + 1) / 2) - 64 * gi);  // orders of this group that exist
        const int part = itm.a ? 1 - (cg >> 1) : cg >> 1;
        if (left < 64) {
#pragma unroll
          for (int k = 0; k < 64; ++k) acc[k] = k < left ? acc[k] : 0.f;
        }
        const long long unit = 2 * ((long long)b * sh.nT + (row0 >> 6)) + (cg & 1);
        const int orow0 = 64 * part + (row0 & 63);
        store_rows64<1, true>(a.out, stage, lane, unit, g, lane, orow0 + lane, true, {unit}, {orow0}, acc);
      } else if constexpr (MODE == kPhiForward) {
        // part cg mod 2 of ring unit cg / 2: 64 rings; P_m or Q_m with K = t.  The even orders of the
        // warp's 32 are 16 rows of one unit, the odd ones 16 rows of another.
        const int per = a.B * sh.nT, part = cg & 1;
        const int un = (int)((cg >> 1) ? itm.u1 : itm.u0) - itm.a * per;
        const int q0 = row0 >> 1, odd = lane & 1;
        const bool has_e = (q0 >> 6) < sh.gE, has_o = (q0 >> 6) < sh.gO;
        if (!has_e || ((cg >> 1) && itm.u1 == itm.u0)) continue;  // the whole warp (gO <= gE)
        const int b = un / sh.nT, tg = un - b * sh.nT, left = L - 64 * tg;
        if (left < 64) {
#pragma unroll
          for (int k = 0; k < 64; ++k) acc[k] = k < left ? acc[k] : 0.f;
        }
        const long long ue = 2 * ((long long)b * sh.G() + (q0 >> 6)) + itm.a, uo = has_o ? ue + 2 * sh.gE : -1;
        const int r0 = 64 * part + (q0 & 63);
        store_rows64<2, false>(a.out, stage, lane, odd ? uo : ue, tg, (lane >> 1) + 16 * odd, r0 + (lane >> 1), !odd || has_o, {ue, uo},
                        {r0, r0}, acc);
      } else if constexpr (MODE == kPhiInverse) {
        // E re, E im, O re, O im of 16 rings; consecutive lanes hold consecutive samples
        if (row >= L) continue;
        const int b = itm.j / sh.nT, t0 = 64 * (itm.j - b * sh.nT) + 16 * cg;
        const long long o = ((long long)b * L + t0) * sh.N;
        float2* fp = a.f + o + row;
        float2* fm = a.f + o + sh.N - 1 - row;
        const bool mirror = row < L - 1;
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          if (t0 + k >= L) break;
          const float er = acc[k], ei = acc[16 + k], odr = acc[32 + k], odi = acc[48 + k];
          if (in_bounds(fp - a.f, a.f_n, kbTorusOut)) *fp = make_float2(er - odi, ei + odr);
          if (mirror && in_bounds(fm - a.f, a.f_n, kbTorusOut)) *fm = make_float2(er + odi, ei - odr);
          fp += sh.N;
          fm += sh.N;
        }
      } else {
        // theta(P) re, im, theta(Q) re, im of 16 orders |m|: H_{+-m} = theta(P) -+ i theta(Q)
        const int b = itm.j / sh.G(), g = itm.j - b * sh.G();
        const int cls = g < sh.gE ? 0 : 1, gi = cls ? g - sh.gE : g;
        const int am0 = 2 * (64 * gi + 16 * cg) + cls;
        const bool tiles = a.to.mode != 0;
        // tiles: the lanes of a 32-K chunk that exists act together (rows past L are zeros)
        if (am0 >= L || (tiles ? row0 >= a.to.nC * 32 : row >= L)) continue;
        // H_{+m} and H_{-m} in acc[k], acc[16 + k] and acc[32 + k], acc[48 + k]; the odd parity carries -i
        const bool live = row < L;
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          const float pr = acc[k], pi = acc[16 + k], qr = acc[32 + k], qi = acc[48 + k];
          const float2 hp = make_float2(pr + qi, pi - qr), hm = make_float2(pr - qi, pi + qr);
          acc[k] = live ? (itm.a ? hp.y : hp.x) : 0.f;
          acc[16 + k] = live ? (itm.a ? -hp.x : hp.y) : 0.f;
          acc[32 + k] = live ? (itm.a ? hm.y : hm.x) : 0.f;
          acc[48 + k] = live ? (itm.a ? -hm.x : hm.y) : 0.f;
        }
        if (!tiles) {
          float2* op = a.f + ((long long)b * sh.N + (am0 + L - 1)) * L + row;
          float2* on = a.f + ((long long)b * sh.N + (L - 1 - am0)) * L + row;
#pragma unroll
          for (int k = 0; k < 16; ++k) {
            if (am0 + 2 * k >= L) break;
            if (in_bounds(op - a.f, a.f_n, kbTorusOut)) *op = make_float2(acc[k], acc[16 + k]);
            if (am0 + 2 * k > 0 && in_bounds(on - a.f, a.f_n, kbTorusOut)) *on = make_float2(acc[32 + k], acc[48 + k]);
            op += 2 * L;
            on -= 2 * L;
          }
          continue;
        }
        // the projection's data tiles (|m|, m' / 32): rows sign * NC/2 + 2b + part, K = m', the negative
        // half carrying (-1)^{m'} (zeros for m = 0; padding rows stay as the plan zeroed them).  The
        // rows' offsets are the same in every tile, the tiles of the 16 orders two |m| apart.
        const int sl = (a.b0 + b) / a.to.Bs, bs = a.b0 + b - sl * a.to.Bs;
        const int half = a.to.NC / 2;
        if (am0 == 0) acc[32] = acc[48] = 0.f;
        const float sgn = (row & 1) ? -1.f : 1.f;
        if (a.to.mode == 2)
          put_orders<true>(a.to, sl, am0, row, lane, L, half, 2 * bs, sgn, acc);
        else
          put_orders<false>(a.to, sl, am0, row, lane, L, half, 2 * bs, sgn, acc);
      }
    }
    if constexpr (MODE == kThetaInverse || MODE == kPhiForward) {
      if (lane == 0) bulk_wait_read<0>();  // the staging memory is read before the CTA leaves
    }
  }
  fence_before();
  __syncthreads();
  if constexpr (PAIR) cluster_sync();  // the pair leaves together: each reads the other's shared memory
  fence_after();
  if (*abort && threadIdx.x == 0) atomicOr(a.status, 2);
  if (warp == 1) {
    if constexpr (PAIR) tmem_dealloc_pair(tbase, 512);
    else tmem_dealloc(tbase, 512);
  }
}

template <int MODE>
__global__ void __launch_bounds__(kThreads, 1) torus_gemm_kernel(const __grid_constant__ TgArgs a) {
  torus_gemm<MODE, false>(a);
}
template <int MODE>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1) torus_gemm_pair_kernel(const __grid_constant__ TgArgs a) {
  torus_gemm<MODE, true>(a);
}

// ---------------------------------------------------------------------------------------------
// Plan-time matrices
// ---------------------------------------------------------------------------------------------
enum Matrix { kCosTheta = 0, kSinTheta, kCosPhiInv, kSinPhiInv, kCosPhiFwd, kSinPhiFwd, kWeightEven, kWeightOdd, kCosAdj, kSinAdj,
              kMatrices };

// Entry (row, k) of matrix `which`.
__device__ double matrix_entry(int which, const Shape& sh, const double2* cs, const double2* T, int row, int k) {
  const int L = sh.L, N = sh.N;
  auto at = [&](int order, int node) { return cs[(int)(((long long)order * (2 * node + 1)) % (2 * N))]; };
  if (row >= L) return 0.0;
  switch (which) {
    case kCosTheta:  // row t, k = m'
      return k >= L ? 0.0 : k == 0 ? 1.0 : 2.0 * at(k, row).x;
    case kSinTheta:
      return k >= L || row == L - 1 ? 0.0 : 2.0 * at(k, row).y;
    case kCosPhiInv:
    case kSinPhiInv: {  // row p, k: even orders first
      const int m = k < 64 * sh.gE ? 2 * k : 2 * (k - 64 * sh.gE) + 1;
      if (m >= L) return 0.0;
      return which == kCosPhiInv ? at(m, row).x : row == L - 1 ? 0.0 : at(m, row).y;
    }
    case kCosPhiFwd:  // row m, k = p
      return k >= L ? 0.0 : at(row, k).x;
    case kSinPhiFwd:
      return k >= L - 1 ? 0.0 : at(row, k).y;
    case kCosAdj:  // row m', k = t
      return k >= L ? 0.0 : row == 0 ? 1.0 : 2.0 * at(row, k).x;
    case kSinAdj:
      return k >= L - 1 ? 0.0 : 2.0 * at(row, k).y;
    default: break;
  }
  // kWeightEven, kWeightOdd: row m', k = t
  return k >= L ? 0.0 : weight_entry(which == kWeightEven, L, cs, T, row, k);
}

// Tiles [i][chunk] of 128 rows x 32 K of one matrix times `scale`, split; a thread writes 8 K of a row.
__global__ void matrix_tiles_kernel(int which, Shape sh, int chunks, double scale, const double2* __restrict__ cs,
                                    const double2* __restrict__ T, uint8_t* __restrict__ out) {
  const long long w = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int per = chunks * 4;  // 8-K pieces of a row
  if (w >= (long long)sh.nI * 128 * per) return;
  const int piece = (int)(w % per), row = (int)(w / per), c = piece >> 2, q = piece & 3;
  uint32_t h[4], l[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    // the parts of the FP64 entry, each rounded to nearest
    const double a = scale * matrix_entry(which, sh, cs, T, row, 8 * piece + 2 * i);
    const double b = scale * matrix_entry(which, sh, cs, T, row, 8 * piece + 2 * i + 1);
    const __half ah = __double2half(a), bh = __double2half(b);
    const __half2 hh = __halves2half2(ah, bh);
    const __half2 ll = __halves2half2(__double2half(a - (double)__half2float(ah)), __double2half(b - (double)__half2float(bh)));
    h[i] = *reinterpret_cast<const uint32_t*>(&hh);
    l[i] = *reinterpret_cast<const uint32_t*>(&ll);
  }
  const int r = row & 127;
  uint8_t* t = out + ((size_t)(row >> 7) * chunks + c) * kUnitBytes;
  *(uint4*)(t + sw128(r, 16 * q)) = make_uint4(h[0], h[1], h[2], h[3]);
  *(uint4*)(t + sw128(r, 64 + 16 * q)) = make_uint4(l[0], l[1], l[2], l[3]);
}

}  // namespace

struct TorusPlan {
  Shape sh{};
  uint8_t* mats = nullptr;  // all matrices, one allocation
  uint8_t* mat[kMatrices] = {};
  int chunks[kMatrices] = {};
  float alpha[kMatrices] = {};
  size_t bytes = 0;
  int sms = 0;
  bool pair = false;
};

// Shared memory of a pass: as many stages as fit beside the staging memory.
static int stage_bytes(int pass, bool pair) {
  return ((pass == kPhiInverse ? 2 : 1) + (pair ? 1 : 2)) * kUnitBytes;
}
static int staging_bytes(int pass) { return pass == kThetaInverse || pass == kPhiForward ? kEpiWarps * kStageWarp : 0; }
static int stages_of(int pass, bool pair) {
  return std::min(kMaxStages, (212 * 1024 - staging_bytes(pass)) / stage_bytes(pass, pair));
}
static size_t smem_of(int pass, bool pair) {
  return (size_t)stages_of(pass, pair) * stage_bytes(pass, pair) + staging_bytes(pass) + 1024;
}

// Units of a pass's data operand and its chunks.
static long long pass_units(const Shape& sh, int pass, int B) {
  return 2ll * B * (pass == kThetaInverse || pass == kThetaForward ? sh.G() : sh.nT);
}
static int pass_chunks(const Shape& sh, int pass) { return pass == kPhiInverse ? sh.nKm() : sh.nKs; }

// Bytes of one field's operand: the largest of the four passes'.
static size_t field_bytes(const Shape& sh) {
  size_t n = 0;
  for (int p = 0; p < 4; ++p) n = std::max(n, operand_bytes(pass_units(sh, p, 1), pass_chunks(sh, p)));
  return n;
}

size_t torus_operand_bytes(const TorusPlan* p, int B) { return field_bytes(p->sh) * B; }

// The passes hold two operands at a time.  As long as these stay within kWhole all fields go at once, one operand in
// place of the half rows (which are read by then).  Beyond that, where a field's operand is the larger
// (padding: 3.9 times at L = 65, 1.5 at L = 257, none from L = 1024 on), the fields run in slices whose operands share
// kSlice bytes, which is thousands of fields at L = 65 and more than a hundred at L = 513, so that every launch still
// fills the GPU: a plan then holds little more than its half rows.  Held by an FP32 plan, all fields at once and in slices:
// L = 65, B = 20000 10.5 and 3.4 GB, L = 300, B = 2000 8.0 and 4.9; inverse and forward 24.8 and 25.0 ms, 113.3 and 113.5.
TorusWork torus_work(int L, int B) {
  constexpr size_t kWhole = 4ull << 30, kSlice = 2ull << 30;
  const Shape sh = make_shape(L);
  const size_t half = (size_t)sh.N * sh.L * sizeof(float2), op = field_bytes(sh);
  TorusWork w;
  if (2 * op * B <= kWhole || 10 * op <= 11 * half) {
    w.fields = B;
    w.w1 = w.w2 = std::max(half, op) * B;
  } else {
    const int most = (int)std::max<size_t>(1, kSlice / (2 * op)), n = (B + most - 1) / most;
    w.fields = (B + n - 1) / n;
    w.w1 = half * B;
    w.w2 = 2 * op * w.fields;
  }
  return w;
}

template <int MODE>
static cudaError_t gemm_attr() {
  cudaError_t e;
  if ((e = prefer_shared(torus_gemm_kernel<MODE>)) != cudaSuccess || (e = prefer_shared(torus_gemm_pair_kernel<MODE>)) != cudaSuccess)
    return e;
  if ((e = cudaFuncSetAttribute(torus_gemm_kernel<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)smem_of(MODE, false))) != cudaSuccess)
    return e;
  return cudaFuncSetAttribute(torus_gemm_pair_kernel<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_of(MODE, true));
}

cudaError_t torus_setup(TorusPlan** out, int L, int device) {
  *out = nullptr;
  TorusPlan* p = new TorusPlan();
  const Shape sh = p->sh = make_shape(L);
  double2* tmp = nullptr;
  cudaError_t e;
  size_t at[kMatrices], total = 0;
  const size_t ncs = 2 * (size_t)sh.N;
  {
    for (int k = 0; k < kMatrices; ++k) {
      p->chunks[k] = (k == kCosPhiInv || k == kSinPhiInv) ? sh.nKm() : sh.nKs;
      at[k] = total;
      total += (size_t)sh.nI * p->chunks[k] * kUnitBytes;
    }
    if ((e = cudaDeviceGetAttribute(&p->sms, cudaDevAttrMultiProcessorCount, device)) != cudaSuccess) goto fail;
    p->pair = sh.nI > 1;
    if ((e = prefer_shared(pack_theta_kernel)) != cudaSuccess || (e = prefer_shared(pack_phi_kernel)) != cudaSuccess) goto fail;
    if ((e = gemm_attr<kThetaInverse>()) != cudaSuccess || (e = gemm_attr<kPhiInverse>()) != cudaSuccess ||
        (e = gemm_attr<kPhiForward>()) != cudaSuccess || (e = gemm_attr<kThetaForward>()) != cudaSuccess)
      goto fail;
    if ((e = dev_malloc(&p->mats, total)) != cudaSuccess) goto fail;
    p->bytes = total;
    if ((e = dev_malloc(&tmp, (ncs + (size_t)L * L) * sizeof(double2))) != cudaSuccess) goto fail;
    double2* T = tmp + ncs;
    node_table_kernel<<<(unsigned)((ncs + 255) / 256), 256>>>(sh.N, tmp);
    weight_prefix_kernel<<<(unsigned)((L + 31) / 32), 32>>>(L, tmp, T);
    // the weight matrices' entries stay below 128 / N^2
    const int ew = 7 + (int)std::floor(2.0 * std::log2((double)sh.N));
    for (int k = 0; k < kMatrices; ++k) {
      p->mat[k] = p->mats + at[k];
      const int ex = (k == kWeightEven || k == kWeightOdd) ? ew : 13;
      p->alpha[k] = std::ldexp(1.f, 14 - ex);
      const long long n = (long long)sh.nI * 128 * p->chunks[k] * 4;
      matrix_tiles_kernel<<<(unsigned)((n + 255) / 256), 256>>>(k, sh, p->chunks[k], std::ldexp(1.0, ex), tmp, T, p->mat[k]);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) goto fail;
    if ((e = cudaDeviceSynchronize()) != cudaSuccess) goto fail;
    cudaFree(tmp);
  }
  *out = p;
  return cudaSuccess;
fail:
  if (tmp) cudaFree(tmp);
  torus_destroy(p);
  return e;
}

void torus_destroy(TorusPlan* p) {
  if (!p) return;
  if (p->mats) cudaFree(p->mats);
  delete p;
}

size_t torus_bytes(const TorusPlan* p) { return p ? p->bytes : 0; }

template <int MODE>
static cudaError_t launch(const TorusPlan* p, TgArgs& a, int s, int B, int col_tiles, int mat, int* status, long long wait_ns,
                          cudaStream_t st) {
  a.sh = p->sh;
  a.s = s;
  a.B = B;
  a.stages = stages_of(MODE, p->pair);
  a.row_tiles = p->pair ? (p->sh.nI + 1) / 2 : p->sh.nI;
  a.ntiles = col_tiles * a.row_tiles;
  a.A[0] = p->mat[mat];
  a.A[1] = p->mat[mat + 1];
  a.a_chunks = p->chunks[mat];
  a.alpha = p->alpha[mat];
  a.status = status;
  a.wait_ns = wait_ns;
  if (p->pair)
    torus_gemm_pair_kernel<MODE><<<2 * std::min(a.ntiles, p->sms / 2), kThreads, smem_of(MODE, true), st>>>(a);
  else
    torus_gemm_kernel<MODE><<<std::min(a.ntiles, p->sms), kThreads, smem_of(MODE, false), st>>>(a);
  return cudaGetLastError();
}

cudaError_t torus_inverse(const TorusPlan* p, int s, int B, const void* F, size_t f_bytes, void* x_work, void* y_work, void* out,
                          size_t out_bytes, int* status, long long wait_ns, cudaStream_t st, int* launches, int step) {
  const Shape& sh = p->sh;
  const Operand x = operand(x_work, pass_units(sh, kThetaInverse, B), sh.nKs);
  const Operand y = operand(y_work, pass_units(sh, kPhiInverse, B), sh.nKm());
  TgArgs a{};
  if (step == 0) {
    const int blocks = ((sh.L + 1) / 2 + 15) / 16 + (sh.L / 2 + 15) / 16;
    pack_theta_kernel<<<dim3((unsigned)(B * blocks), (unsigned)((sh.nKs / 2 + 1) / 2)), 512, 0, st>>>(sh, B, (const float2*)F, x, (long long)(f_bytes / sizeof(float2)));
    a.in = x;
    a.out = y;
    *launches += 2;
    return launch<kThetaInverse>(p, a, s, B, B * sh.G(), kCosTheta, status, wait_ns, st);
  }
  a.in = y;
  a.f = (float2*)out;
  a.f_n = (long long)(out_bytes / sizeof(float2));
  *launches += 1;
  return launch<kPhiInverse>(p, a, s, B, B * sh.nT, kCosPhiInv, status, wait_ns, st);
}

cudaError_t torus_analysis(const TorusPlan* p, int adjoint, int s, int B, const void* f, size_t f_bytes, void* x_work, void* y_work,
                           void* H, size_t h_bytes, const TileOut* tiles, int b0, int* status, long long wait_ns, cudaStream_t st,
                           int* launches, int step) {
  const Shape& sh = p->sh;
  const Operand x = operand(x_work, pass_units(sh, kPhiForward, B), sh.nKs);
  const Operand y = operand(y_work, pass_units(sh, kThetaForward, B), sh.nKs);
  TgArgs a{};
  if (step == 0) {
    pack_phi_kernel<<<dim3((unsigned)(B * ((sh.L + 15) / 16)), (unsigned)((sh.nKs / 2 + 1) / 2)), 512, 0, st>>>(sh, B, (const float2*)f, x, (long long)(f_bytes / sizeof(float2)));
    a.in = x;
    a.out = y;
    *launches += 2;
    return launch<kPhiForward>(p, a, s, B, 2 * ((B * sh.nT + 1) / 2), kCosPhiFwd, status, wait_ns, st);
  }
  a.in = y;
  a.b0 = b0;
  if (tiles) a.to = *tiles;
  a.f = (float2*)H;
  a.f_n = (long long)(h_bytes / sizeof(float2));
  *launches += 1;
  return launch<kThetaForward>(p, a, s, B, B * sh.G(), adjoint ? kCosAdj : kWeightEven, status, wait_ns, st);
}

SSHT_BOUNDS_TU(torus_pass)

}  // namespace ssht
