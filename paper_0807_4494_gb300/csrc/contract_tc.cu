// The O(L^3) contractions on the tcgen05 tensor cores (split FP16 or BF16 products, FP32 accumulation
// in tensor memory), for batched transforms.
//
// For each m >= 0 both signs of m share one matrix (eqn wignerd_sym6 gives
// Delta^l_{m',-m} = (-1)^{l+m'} Delta^l_{m'm}):
//   A_m[m', l] = U_l[m'] Delta^l_{m'm},   U_l[m'] = sqrt((2l+1)/4pi) Delta^l_{m',-s},
// nonzero for l >= max(m, m', |s|).  With columns j = (sign, part, b) over 4B real columns:
//   inverse (eqn fourier_coeff):  D[m', j] = sum_l A_m[m', l] V_m[l, j],
//       V_m[l, (0, part, b)] = part(sf_{l,m}[b]),  V_m[l, (1, part, b)] = (-1)^l part(sf_{l,-m}[b]);
//       F_{m m'} = (-1)^s i^{-(m+s)} D[m', (0, ., b)],  F_{-m, m'} = (-1)^s i^{m-s} (-1)^{m'} D[m', (1, ., b)].
//   forward / adjoint projection:  P[l, j] = sum_{m'} A_m[m', l] Y_m[m', j],
//       Y_m[m', (0, part, b)] = part(H_{m m'}[b]),  Y_m[m', (1, part, b)] = (-1)^{m'} part(H_{-m m'}[b]);
//       sf_{lm} = (-1)^s i^{m+s} P[l, (0, ., b)],  sf_{l,-m} = (-1)^s i^{-m+s} (-1)^l P[l, (1, ., b)].
// So every m is a real GEMM with M = 128-row blocks of m' (inverse) or l (forward), K = l or m'
// in chunks of 32, N = 2H columns, H = 2B rounded up to 16 (column sign*H + 2b + part).
//
// Split forms.  SSHT_TF32X3 plans: x = hi + lo in two parts of 11 significant bits and the product
// hi*hi + hi*lo + lo*hi (the dropped lo*lo is ~2^-24 relative), the arithmetic of a 3xTF32 split with the parts
// held as FP16, which the tensor cores multiply at twice the TF32 rate and which take half the bytes.  FP16's
// range is met by powers of two: 2^10 for A (|U Delta| < 18.1), for the data one a (row pair, chunk) -- a
// field's real and imaginary part over 32 K -- from its largest magnitude, undone when the segment is added.
// SSHT_BF16X6 plans: three BF16 parts, the six products down to 2^-24.
//
// Accumulation.  The tensor core's FP32 accumulation truncates (rounds toward zero); over the
// accumulation steps of K = 1024 that bias alone reaches ~1e-5 relative.  So each K chunk
// accumulates into a fresh tensor-memory segment, the small correction products first and the
// large ones last (truncation then acts on two large steps only), and the epilogue warps
// add every segment into FP32 running sums in registers (round to nearest).
//
// Operands are written once per call (A also once per plan with the Delta cache) as tiles of split parts
// already in the K-major SWIZZLE_128B layout (split-FP16: 128 bytes a row and 32 K, as many as FP32 values),
// so that the main kernel moves them with 1-D bulk copies.  Main kernel: persistent, one CTA per SM, five
// warpgroups: warp 0 issues the bulk copies (a ring of 2-4 stages), warp 1 issues tcgen05.mma into one of two
// 128 x 256 FP32 accumulator segments in tensor memory (both as whole warps with an elected lane: a single
// lane's loop took 70 clocks a product), sixteen warps (four per 32-lane quarter of tensor memory, each
// every fourth group of 16 columns) read the accumulator with tcgen05.ld, apply the phases and write the
// outputs (the inverse writes half rows m' >= 0 of F; the torus passes apply the extension).  Work items (m,
// row block) are sorted (groups of four m, or decreasing length) and dealt to the CTAs by a greedy
// schedule made on the host (schedule()).  Every wait is bounded; a
// timeout latches a status bit and the CTA drains its copies and MMAs before leaving.
#include "ssht_internal.h"
#include "bounds.cuh"
#include "f32_round.h"
#include "tc_common.cuh"

#include <algorithm>
#include <queue>
#include <vector>

namespace ssht {
namespace {

using namespace tc;

constexpr int TM = kTileRows;              // rows per tile
constexpr int TK = kTileK;                 // K per chunk (two FP16 parts: 128 bytes a row)
constexpr int A_PART = kAPart;             // 16 KB: one part of an A tile
constexpr int MAX_STAGES = 4;             // pipeline depth: a plan parameter, 2 .. MAX_STAGES
constexpr int SCALE_SLOTS = 8;            // ring of the chunks' scales (MAX_STAGES + 2 would do)
constexpr int EPI_WARPS = 16;                      // four per tensor-memory lane quarter
// producer, MMA and two idle warps, then the epilogue's; 96 registers a thread at launch, of which the
// first warpgroup gives some up for the epilogue's 64 running sums
constexpr int THREADS = 128 + 32 * EPI_WARPS;
constexpr int REGS_ISSUE = 32, REGS_EPILOGUE = 112;
static_assert(128 * REGS_ISSUE + 32 * EPI_WARPS * REGS_EPILOGUE <= THREADS * 96, "register shares");

__host__ __device__ inline long long tri_ll(long long m) { return m * (m + 1) / 2; }
__host__ __device__ inline size_t doff(long long l) { return (size_t)(l * (l + 1) * (2 * l + 1) / 6); }

struct Item {
  int m, i, c0, c1;     // row block i of m; K chunks [c0, c1)
  long long atile;      // index of the A tile of chunk c0
};

struct TcArgs {
  int L, s, B, Bs, NC;    // Bs: fields of a slice (blockIdx.y); NC = 2H: padded columns, H = 2 Bs rounded up to 16 (<= 128)
  int stages;             // pipeline depth
  const int* sched;       // CTA b runs items [sched[b], sched[b + 1]) in order
  const Item* items;
  const uint8_t* A;       // packed A tiles
  const uint8_t* X;       // packed data tiles, xslice bytes a slice
  size_t xslice;
  const float* XS;        // split-FP16: their scales, [tile][NC / 2]
  const long long* xoff;  // per m: data tile index of chunk xc0(m)
  const int* xc0;         // per m: first chunk stored for m
  float2* out;            // half rows [B][N][L] (rows by signed order; inverse: F, columns m'; forward with
                          // `rows`: columns l >= |m|), or flm [B][L*L]
  int rows;               // forward: half rows instead of flm
  int* status;
  long long wait_ns;      // spin limit of the pipeline waits
  long long a_tiles, x_tiles;  // extents of A and of a slice's data tiles (index checks)
  long long out_field;         // elements of a field in out
};

__device__ __forceinline__ float2 ipow_signed(int s, int k) {
  const int r = ((k % 4) + 4) % 4;
  float a = (r == 0) ? 1.f : (r == 2) ? -1.f : 0.f;
  float b = (r == 1) ? 1.f : (r == 3) ? -1.f : 0.f;
  if (s & 1) { a = -a; b = -b; }
  return make_float2(a, b);
}

// ---------------------------------------------------------------------------------------------
// Packing: A tiles from the FP64 Delta table
// ---------------------------------------------------------------------------------------------

// Inverse A tile (m, i, c): rows m' = 128 i + r, columns l = 32 c + k (K-major).
// Forward A tile (m, i, c): rows l = 128 i + r, columns m' = 32 c + k.
// Every thread issues its 16 table loads before converting any of them.
template <bool FWD, bool BF>
__global__ void __launch_bounds__(256) pack_a_kernel(int L, int s, const Item* __restrict__ items,
                                                     const double* __restrict__ table, const float* __restrict__ Uf,
                                                     uint8_t* __restrict__ A, long long a_tiles) {
  __shared__ __align__(16) uint8_t tile[kParts<BF> * A_PART];
  constexpr int PER = TM * TK / 256;
  const Item it = items[blockIdx.y];
  const int c = it.c0 + blockIdx.x;
  if (c >= it.c1) return;
  const int m = it.m, Lp = L - 1, as = s < 0 ? -s : s;
  double d[PER];
  float u[PER];
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    const int e = threadIdx.x + q * 256;
    const int r = FWD ? e / TK : e % TM, k = FWD ? e % TK : e / TM;
    const int rowv = it.i * TM + r, colv = c * TK + k;
    const int mp = FWD ? colv : rowv, l = FWD ? rowv : colv;
    const bool ok = l <= Lp && mp <= Lp && l >= m && l >= mp && l >= as;
    // Delta^l_{m' m} = (-1)^{m'-m} Delta^l_{m m'}: row m of degree l, contiguous in m'
    const long long ti = (long long)doff(l) + (long long)m * (l + 1) + mp, ui = (long long)tri_ll(l) + mp;
    d[q] = (ok && in_bounds(ti, (long long)doff(L), kbPackAIn)) ? __ldg(&table[ti]) : 0.0;
    u[q] = (ok && in_bounds(ui, (long long)tri_ll(L), kbPackAIn)) ? __ldg(&Uf[ui]) : 0.f;
  }
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    const int e = threadIdx.x + q * 256;
    const int r = FWD ? e / TK : e % TM, k = FWD ? e % TK : e / TM;
    const int mp = FWD ? c * TK + k : it.i * TM + r;
    const float a = u[q] * f64_to_f32_rn(d[q]);
    put_parts<BF>(tile, A_PART, sw128(r, 2 * k), ((mp - m) & 1) ? -a : a);
    if (BF) *(uint16_t*)(tile + A_PART + (sw128(r, 2 * k) ^ 64u)) = 0;
  }
  __syncthreads();
  if (!in_bounds(it.atile + blockIdx.x, a_tiles, kbPackAOut)) return;
  constexpr int GA = kParts<BF> * A_PART;  // bytes of a tile in global memory
  uint4* dst = (uint4*)(A + (size_t)(it.atile + blockIdx.x) * GA);
  const uint4* src = (const uint4*)tile;
  for (int e = threadIdx.x; e < GA / 16; e += blockDim.x) dst[e] = src[e];
}

// ---------------------------------------------------------------------------------------------
// Packing: data tiles (rows j = (sign, part, b), K-major over 32 l or m')
// ---------------------------------------------------------------------------------------------

// Inverse data tiles (m, c): V_m[l, j], l = 32 c + k, rows j = sign * NC/2 + 2b (real part) and
// 2b + 1 (imaginary part), for 16 consecutive m at once.  For two fields at a time the coefficients
// sf_{l,+-m} of the 32 degrees of chunk c are read as runs of 16 consecutive orders (coalesced)
// and turned around in shared memory.  Split-FP16: a thread then takes
// 8 K of one order, sign and field, four neighbouring threads the 32 K of a tile row, so that they find the
// row pair's power of two with two shuffles and store 16 bytes at a time.  Split-BF16: a warp takes a row
// pair, a lane one K.  The rows of padding fields stay as tc_configure zeroed them.  Fields run in slices of Bs, slice z
// in its own tile region of xslice bytes, and a CTA takes `per` fields of a slice, an even number
// (blockIdx.z: slice and group of fields): eight, or two where that leaves SMs without a CTA.  Bound by HBM
// traffic (1.1 GB at L = 1024, B = 64: 0.16 ms) and by how many loads are in flight: six CTAs on an SM (40
// registers) take 0.28 ms where three with the next fields' loads under way (80 registers) took 0.47 and
// a CTA of 64 KB staging with bulk stores 0.66; at L = 512, B = 32 42 us, 68 before.

template <bool BF>
__global__ void __launch_bounds__(256, 6) pack_v_kernel(int L, int s, int Btot, int Bs, int per, size_t xslice, int NC,
                                                     const int* __restrict__ xc0, const long long* __restrict__ xoff,
                                                     const float2* __restrict__ flm, uint8_t* __restrict__ X,
                                                     float* __restrict__ XS) {
  __shared__ float2 sv[2][32][33];
  const int half = NC / 2, groups = (Bs + per - 1) / per, z = blockIdx.z / groups, bg = (blockIdx.z - z * groups) * per;
  const int B = min(Bs, Btot - z * Bs);
  const long long flm_n = (long long)Btot * L * L, flm0 = (long long)z * Bs * L * L;
  const long long x_tiles = (long long)(xslice / (kParts<BF> * (size_t)NC * 128));
  X += (size_t)z * xslice;
  if (!BF) XS += (size_t)z * x_tiles * half;
  const int c = blockIdx.x, m0 = 16 * blockIdx.y;
  // xc0 grows with m: when chunk c is below the first stored chunk of m0, no tile of this CTA's 16
  // orders is stored (about half the grid: the degrees of chunk c all lie below m0)
  if (m0 >= L || c < xc0[m0] || bg >= B) return;
  const int as = s < 0 ? -s : s;
  const int part_bytes = NC * 128;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int b_end = min(bg + per, B);
  // 32 degrees l x (orders m0 .. m0 + 15, then -m0 .. -m0 - 15) of a field: four values a thread, whose
  // places in a field are the same for every field
  int at[4];
  unsigned have = 0, neg = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int q = threadIdx.x + 256 * i, lo = q >> 5, col = q & 31, sign = col >> 4, m = m0 + (col & 15);
    const int l = c * TK + lo;
    at[i] = l * l + l + (sign ? -m : m);
    if (m < L && l < L && l >= m && l >= as && !(sign && m == 0)) have |= 1u << i;
    if (sign && (l & 1)) neg |= 1u << i;
  }
  for (int b = bg; b < b_end; b += 2) {
#pragma unroll
    for (int f = 0; f < 2; ++f) {
      const long long f0 = flm0 + (long long)(b + f) * L * L;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int q = threadIdx.x + 256 * i;
        float2 x = make_float2(0.f, 0.f);
        if (((have >> i) & 1u) && b + f < B && in_bounds(f0 + at[i], flm_n, kbPackVIn)) x = __ldg(&flm[f0 + at[i]]);
        sv[f][q >> 5][q & 31] = ((neg >> i) & 1u) ? make_float2(-x.x, -x.y) : x;
      }
    }
    __syncthreads();
    if constexpr (BF) {
      for (int cb = warp; cb < 64; cb += 8) {
        const int f = cb >> 5, sign = (cb >> 4) & 1, m = m0 + (cb & 15), j = sign * half + 2 * (b + f);
        if (m >= L || c < xc0[m] || b + f >= b_end) continue;  // tile (m, c) is not stored
        const long long tix = xoff[m] + (c - xc0[m]);
        if (!in_bounds(tix, x_tiles, kbPackVOut) || !in_bounds(j + 1, NC, kbPackVOut)) continue;
        const float2 x = sv[f][lane][cb & 31];
        put_rows2<BF>(X + (size_t)tix * kParts<BF> * part_bytes, part_bytes, j, lane, x.x, x.y, 1.f, true);
      }
    } else {
      const int f = warp >> 2, cb = (warp & 3) * 8 + (lane >> 2), kq = lane & 3;
      const int sign = cb >> 4, m = m0 + (cb & 15), j = sign * half + 2 * (b + f);
      float x[8], y[8], amax = 0.f;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const float2 w = sv[f][8 * kq + k][cb];
        x[k] = w.x;
        y[k] = w.y;
        amax = fmaxf(amax, fmaxf(fabsf(w.x), fabsf(w.y)));
      }
      amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 1));
      amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 2));
      float sc;
      const float up = block_power(amax, &sc);
      if (m < L && c >= xc0[m] && b + f < b_end) {
        const long long tix = xoff[m] + (c - xc0[m]);
        if (in_bounds(tix, x_tiles, kbPackVOut) && in_bounds(j + 1, NC, kbPackVOut)) {
          uint8_t* tile = X + (size_t)tix * part_bytes;
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const float* w = i ? y : x;
            uint4 h, l;
            split2(up * w[0], up * w[1], &h.x, &l.x);
            split2(up * w[2], up * w[3], &h.y, &l.y);
            split2(up * w[4], up * w[5], &h.z, &l.z);
            split2(up * w[6], up * w[7], &h.w, &l.w);
            const uint32_t off = sw128(j + i, 16 * kq);
            *(uint4*)(tile + off) = h;
            *(uint4*)(tile + (off ^ 64u)) = l;
          }
          if (kq == 0) XS[(size_t)tix * half + (j >> 1)] = sc;
        }
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------------------------
// The tensor-core GEMM
// ---------------------------------------------------------------------------------------------

template <bool FWD, bool BF>
__global__ void __launch_bounds__(THREADS, 1) tc_gemm_kernel(TcArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  constexpr int GA = kParts<BF> * A_PART;  // bytes of an A tile
  const int b_part = a.NC * 128;
  const int gx = kParts<BF> * b_part;      // bytes of a data tile
  const int stage_bytes = GA + gx;
  const int STAGES = a.stages;
  __shared__ __align__(8) uint64_t full[MAX_STAGES], empty[MAX_STAGES], seg_full[2], seg_empty[2], done_bar;
  // split-FP16: the chunks' scales, filled ahead of the products.  Slot reuse needs no barrier: when the
  // producer fills chunk n, chunk n - STAGES has been multiplied, so the epilogue has released chunk
  // n - STAGES - 2 and read the scales of the chunk before that.
  __shared__ __align__(16) float scales[SCALE_SLOTS][128];
  __shared__ __align__(8) uint64_t scale_full[SCALE_SLOTS];
  static_assert(SCALE_SLOTS > MAX_STAGES + 2 && (SCALE_SLOTS & (SCALE_SLOTS - 1)) == 0, "scale ring");
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag;
  // this slice's outputs and fields (read again for every item: kept in registers, they cost the sums' loop some)
  __shared__ float2* slice_out;
  __shared__ int slice_fields;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp == 1) tmem_alloc(&tmem_base, 512);
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int k = 0; k < 2; ++k) {
      mbar_init(&seg_full[k], 1);
      mbar_init(&seg_empty[k], EPI_WARPS);
    }
    for (int k = 0; k < SCALE_SLOTS; ++k) mbar_init(&scale_full[k], 1);
    mbar_init(&done_bar, 1);
    abort_flag = 0;
    const int first = blockIdx.y * a.Bs;
    slice_out = a.out + first * a.out_field;
    slice_fields = min(a.Bs, a.B - first);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tbase = tmem_base;
  volatile int* abort = &abort_flag;
  const int nC = (a.L + TK - 1) / TK;
  const int w_begin = a.sched[blockIdx.x], w_end = a.sched[blockIdx.x + 1];

  if (warp < 4) {
    regs_dec<REGS_ISSUE>();
    if (warp == 0) {
      // ---- producer: bulk copies of the A and data tiles of every chunk ----
      const bool one = elect_one();
      int s = 0, ph = 1, n = 0;     // stage, parity its empty barrier is waited for, chunk
      uint32_t used = 0, uph = 0;   // stages that were filled, and the parity of their last fill
      const uint8_t* X = a.X + (size_t)blockIdx.y * a.xslice;
      const float* XS = BF ? nullptr : a.XS + (size_t)blockIdx.y * a.x_tiles * (a.NC / 2);
      for (int w = w_begin; w < w_end && !*abort; ++w) {
        const Item itm = a.items[w];
        const long long x0 = FWD ? (long long)itm.m * nC : a.xoff[itm.m] - a.xc0[itm.m];
        for (int c = itm.c0; c < itm.c1; ++c, ++n) {
          if (!__all_sync(0xffffffffu, mbar_wait(&empty[s], ph, abort, a.wait_ns))) {
            *abort = 1;
            break;
          }
          if (one) {
            // a tile index outside its array is recorded and tile 0 copied instead (the pipeline
            // still completes; the result is wrong and the record says why)
            const long long at = itm.atile + (c - itm.c0);
            const uint8_t* asrc = in_bounds(at, a.a_tiles, kbGemmA) ? a.A + (size_t)at * GA : a.A;
            long long xt = x0 + c;
            if (!in_bounds(xt, a.x_tiles, kbGemmX)) xt = 0;
            uint8_t* st = smem + s * stage_bytes;
            if constexpr (!BF) {
              const int slot = n & (SCALE_SLOTS - 1);
              mbar_expect_tx(&scale_full[slot], (uint32_t)(2 * a.NC));
              bulk_g2s(scales[slot], XS + (size_t)xt * (a.NC / 2), (uint32_t)(2 * a.NC), &scale_full[slot]);
            }
            mbar_expect_tx(&full[s], (uint32_t)(GA + gx));
            bulk_g2s(st, asrc, GA, &full[s]);
            bulk_g2s(st + GA, X + (size_t)xt * gx, (uint32_t)gx, &full[s]);
          }
          used |= 1u << s;
          uph = (uph & ~(1u << s)) | ((uint32_t)(ph ^ 1) << s);
          if (++s == STAGES) {
            s = 0;
            ph ^= 1;
          }
        }
      }
      // drain: every issued copy must have landed before the CTA leaves
      for (int k = 0; k < STAGES; ++k)
        if ((used >> k) & 1u) mbar_wait(&full[k], (uph >> k) & 1u, nullptr, kDrainNs);
      if constexpr (!BF)
        for (int k = max(0, n - SCALE_SLOTS); k < n; ++k)
          mbar_wait(&scale_full[k & (SCALE_SLOTS - 1)], (k / SCALE_SLOTS) & 1, nullptr, kDrainNs);
    } else if (warp == 1) {
      // ---- MMA issuer: one tensor-memory segment per chunk, corrections first ----
      const uint32_t idesc = BF ? idesc_bf16(TM, a.NC) : idesc_f16(TM, a.NC);
      const bool one = elect_one();
      const uint32_t lo0 = (smem_u32(smem) >> 4) + kDescLow;
      int s = 0, ph = 0, seg = 0, sph = 1;
      for (int w = w_begin; w < w_end && !*abort; ++w) {
        const int nc = a.items[w].c1 - a.items[w].c0;
        for (int c = 0; c < nc; ++c) {
          const bool here = mbar_wait(&seg_empty[seg], sph, abort, a.wait_ns) && mbar_wait(&full[s], ph, abort, a.wait_ns);
          if (!__all_sync(0xffffffffu, here)) {
            *abort = 1;
            break;
          }
          fence_after();
          if (one) {
            const uint32_t dt = tbase + (uint32_t)(seg * 256);
            const uint32_t la = lo0 + (uint32_t)(s * (stage_bytes >> 4)), lb = la + (GA >> 4);
            if constexpr (BF) {
              // parts h, m at bytes 0 and 64 of part 0, l at byte 0 of part 1; K = 16 (32 bytes)
              // per instruction.  Products from the smallest up: h*l, l*h, m*m, h*m, m*h, h*h.
              const uint32_t oa[3] = {0u, 4u, (uint32_t)(A_PART >> 4)}, ob[3] = {0u, 4u, (uint32_t)(b_part >> 4)};
              const int pa[6] = {0, 2, 1, 0, 1, 0}, pb[6] = {2, 0, 1, 1, 0, 0};
#pragma unroll
              for (int q = 0; q < 6; ++q)
#pragma unroll
                for (int kk = 0; kk < 2; ++kk)
                  mma_f16_lo<false>(dt, la + oa[pa[q]] + 2 * kk, lb + ob[pb[q]] + 2 * kk, idesc, (q | kk) ? 1u : 0u);
            } else {
              // hi at byte 0, lo at byte 64 of a row: hi*lo, lo*hi, hi*hi
#pragma unroll
              for (int q = 0; q < 3; ++q)
#pragma unroll
                for (int kk = 0; kk < 2; ++kk)
                  mma_f16_lo<false>(dt, la + (q == 1 ? 4u : 0u) + 2 * kk, lb + (q == 0 ? 4u : 0u) + 2 * kk, idesc, (q | kk) ? 1u : 0u);
            }
            mma_commit(&empty[s]);
            mma_commit(&seg_full[seg]);
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
      if (one) mma_commit(&done_bar);
      __syncwarp();
      mbar_wait(&done_bar, 0, nullptr, kDrainNs);  // every issued MMA has completed
    }
  } else {
    // ---- epilogue: running sums of the segments, then phases and outputs ----
    regs_inc<REGS_EPILOGUE>();
    const int q = warp & 3;            // tensor-memory lane quarter this warp may access
    const int cg = (warp - 4) >> 2;    // of the NC / 16 groups of 16 columns: cg, cg + 4, cg + 8, cg + 12
    const int r = q * 32 + lane;
    const int L = a.L, Lp = L - 1, NT = 2 * L - 1, s = a.s;
    const int H = a.NC / 2;
    const uint32_t tq = tbase + ((uint32_t)(q * 32) << 16);
    int seg = 0, sph = 0, n = 0;
    for (int w = w_begin; w < w_end && !*abort; ++w) {
      const Item itm = a.items[w];
      float acc[64];
#pragma unroll
      for (int k = 0; k < 64; ++k) acc[k] = 0.f;
      bool ok = true;
      for (int c = itm.c0; c < itm.c1; ++c, ++n) {
        const int slot = n & (SCALE_SLOTS - 1);
        if ((!BF && !mbar_wait(&scale_full[slot], (n / SCALE_SLOTS) & 1, abort, a.wait_ns)) ||
            !mbar_wait(&seg_full[seg], sph, abort, a.wait_ns)) {
          *abort = 1;
          ok = false;
          break;
        }
        fence_after();
        const uint32_t ts = tq + (uint32_t)(seg * 256);
#pragma unroll
        for (int g = 0; g < 4; g += 2) {
          uint32_t v[32];
          const int j = 16 * (4 * g + cg);  // the groups' first columns: j and j + 64
          if (j < a.NC) tmem_ld16_nowait(ts + j, v);
          if (j + 64 < a.NC) tmem_ld16_nowait(ts + j + 64, v + 16);
          tmem_wait_ld();
          if (g == 2) {  // the segment is read: free it before the last sums
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&seg_empty[seg]);
          }
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            if (j + 64 * i >= a.NC) continue;
            if constexpr (BF) {
#pragma unroll
              for (int k = 0; k < 16; ++k) acc[16 * (g + i) + k] += __uint_as_float(v[16 * i + k]);
            } else {
              const float4 s0 = *(const float4*)&scales[slot][(j + 64 * i) / 2], s1 = *(const float4*)&scales[slot][(j + 64 * i) / 2 + 4];
              const float sc[8] = {s0.x, s0.y, s0.z, s0.w, s1.x, s1.y, s1.z, s1.w};
#pragma unroll
              for (int k = 0; k < 16; ++k)
                acc[16 * (g + i) + k] = fmaf(__uint_as_float(v[16 * i + k]), sc[k >> 1], acc[16 * (g + i) + k]);
            }
          }
        }
        seg ^= 1;
        if (seg == 0) sph ^= 1;
      }
      if (!ok) break;
      const int m = itm.m;
      const int rowv = itm.i * TM + r;  // m' (inverse) or l (forward)
      const bool valid = FWD ? (rowv <= Lp && rowv >= m) : (rowv <= Lp);
      if (!valid) continue;
      const int B = *(volatile int*)&slice_fields;
      float2* const out = *(float2* volatile*)&slice_out;
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        const int j = 16 * (4 * g + cg);
        if (j >= a.NC) break;
        const int h = j >= H ? 1 : 0, b0 = (j - h * H) >> 1;  // the sign of m and the first of the group's 8 fields
        if (h == 1 && m == 0) break;
        const int mm = h ? -m : m;
        // the phase, (-1)^{m'} (inverse) or (-1)^l (forward) for -m, and split-FP16's 2^14 / 2^10
        const float2 pu = FWD ? ipow_signed(s, mm + s) : ipow_signed(s, -(mm + s));
        const float rs = ((h && (rowv & 1)) ? -1.f : 1.f) * (BF ? 1.f : 16384.f / kAScale);
        const float2 pz = make_float2(rs * pu.x, rs * pu.y);
        const bool flat = FWD && !a.rows;
        const long long ob = flat ? (long long)L * L : (long long)NT * L;
        const long long o0 = flat ? (long long)rowv * rowv + rowv + mm : (long long)(mm + Lp) * L + rowv;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int b = b0 + k;
          if (b >= B) break;
          const float xr = acc[16 * g + 2 * k], xi = acc[16 * g + 2 * k + 1];
          const long long o = o0 + b * ob;
          if (in_bounds(o, B * a.out_field, kbGemmOut)) out[o] = make_float2(pz.x * xr - pz.y * xi, pz.x * xi + pz.y * xr);
        }
      }
    }
  }
  fence_before();
  __syncthreads();
  fence_after();
  if (*abort && threadIdx.x == 0) atomicOr(a.status, 2);
  if (warp == 1) tmem_dealloc(tbase, 512);
}

// Forward output: half rows P [b][m + Lp][l], l >= |m|, -> flm [b][l^2 + l + m], by 32 x 32 blocks through
// shared memory (both sides in runs of 256 bytes).  blockIdx.x: block of l, y: block of m + Lp, z: field.
__global__ void __launch_bounds__(256) rows_to_flm_kernel(int L, const float2* __restrict__ P, float2* __restrict__ flm,
                                                          long long p_n, long long out_n) {
  __shared__ float2 sv[32][33];
  const int Lp = L - 1, N = 2 * L - 1, l0 = 32 * blockIdx.x, r0 = 32 * blockIdx.y;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  // no entry of the block has l >= |m|
  const int l1 = min(l0 + 31, Lp), m_lo = r0 - Lp, m_hi = min(r0 + 31, N - 1) - Lp;
  if (m_lo > l1 || m_hi < -l1) return;
  const long long pb = (long long)blockIdx.z * N * L, fb = (long long)blockIdx.z * L * L;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int r = r0 + ty + 8 * k, l = l0 + tx, m = r - Lp;
    if (r < N && l < L && l >= m && l >= -m && in_bounds(pb + (long long)r * L + l, p_n, kbGemmOut))
      sv[ty + 8 * k][tx] = P[pb + (long long)r * L + l];
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int l = l0 + ty + 8 * k, r = r0 + tx, m = r - Lp;
    const long long o = fb + (long long)l * l + l + m;
    if (r < N && l < L && l >= m && l >= -m && in_bounds(o, out_n, kbGemmOut)) flm[o] = sv[tx][ty + 8 * k];
  }
}

}  // namespace

// ---------------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------------

struct TcPlan {
  int L = 0, s = 0, B = 0, NC = 0, nC = 0, nI = 0;
  bool bf16 = false;  // split-BF16 (3 parts, 6 products) instead of split-FP16
  TcConfig cfg;
  int Bs = 0, nS = 0;        // fields per slice and slices
  size_t xslice = 0;         // bytes of one slice's data tiles
  std::vector<Item> inv_h, fwd_h;  // work items in creation order (re-sorted by the configuration)
  Item* items_inv = nullptr;  // in schedule order: CTA-major
  Item* items_fwd = nullptr;
  int* sched_inv = nullptr;   // per CTA: first item (grid + 1 entries)
  int* sched_fwd = nullptr;
  int grid_inv = 0, grid_fwd = 0;
  int n_inv = 0, n_fwd = 0;
  long long tiles_A = 0, tiles_inv = 0, xtiles_inv = 0, xtiles_fwd = 0;
  // Forward A tiles (m, i, c): rows l = 128 i + r, K = m' = 32 c + k, tile index abase[m] +
  // 2i(i+1) - 2 i_m(i_m+1) + c with i_m = m / 128 (each (m, i), i >= i_m, holds 4i + 4 slots;
  // entries nothing writes stay zero).  Inverse A tiles A_inv (m, i, c): rows m' = 128 i + r,
  // K = l = 32 c + k, at the item's tile index.  Both are shared by every slice of fields.
  uint8_t* A = nullptr;
  uint8_t* A_inv = nullptr;
  long long* abase = nullptr;
  long long* ibase = nullptr;  // [m * nI + i]: tile index of chunk kc of inverse item (m, i) is ibase + kc
  uint8_t* X = nullptr;        // data tiles, nS slices of xslice bytes
  size_t xbytes = 0;
  float* XS = nullptr;         // split-FP16: scales of the data tiles, nS slices of [tile][NC / 2]
  size_t xsbytes = 0;
  long long* xoff = nullptr;
  int* xc0 = nullptr;
  size_t bytes = 0;
  int grid = 0;
  size_t smem = 0;
  int smem_max = 0;
};

static cudaError_t tc_alloc(void** p, size_t bytes, size_t* total) {
  cudaError_t e = dev_malloc(p, bytes ? bytes : 16);
  if (e == cudaSuccess) *total += bytes;
  return e;
}

template <class K>
static cudaError_t gemm_attrs(K kernel, int bytes) {
  cudaError_t e = prefer_shared(kernel);
  return e != cudaSuccess ? e : cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

static int nc_of(int Bs) { return 2 * (((2 * Bs + 15) / 16) * 16); }
static size_t stage_bytes_of(int NC, bool bf16) { return (bf16 ? 2 : 1) * ((size_t)A_PART + (size_t)NC * 128); }

bool tc_config_fits(const TcPlan* p, const TcConfig& c) {
  if (c.slice < 1 || c.slice > 64 || c.stages < 2 || c.stages > MAX_STAGES) return false;
  const int Bs = std::min(c.slice, p->B);
  return (size_t)c.stages * stage_bytes_of(nc_of(Bs), p->bf16) + 1024 <= (size_t)p->smem_max;
}

// Assign the items, in list order, each to the CTA that becomes free first, with a cost of its
// chunk count plus a fixed share for its epilogue: the schedule a shared work counter would give,
// made on the host.  Items next to each other in the list then run at about the same time on
// different SMs, so that the data tiles they share are read from HBM about once, and the longest
// CTA finishes close to the mean.  Uploads the items CTA-major and the per-CTA offsets.
static cudaError_t schedule(const std::vector<Item>& items, int grid, Item* d_items, int* d_sched) {
  constexpr long long kEpilogueChunks = 2;
  std::priority_queue<std::pair<long long, int>, std::vector<std::pair<long long, int>>, std::greater<>> free_at;
  for (int b = 0; b < grid; ++b) free_at.push({0, b});
  std::vector<std::vector<int>> per(grid);
  for (int w = 0; w < (int)items.size(); ++w) {
    const auto top = free_at.top();
    free_at.pop();
    per[top.second].push_back(w);
    free_at.push({top.first + (items[w].c1 - items[w].c0) + kEpilogueChunks, top.second});
  }
  std::vector<Item> out;
  std::vector<int> start(grid + 1, 0);
  out.reserve(items.size());
  for (int b = 0; b < grid; ++b) {
    start[b] = (int)out.size();
    for (int w : per[b]) out.push_back(items[w]);
  }
  start[grid] = (int)out.size();
  cudaError_t e = cudaMemcpy(d_items, out.data(), out.size() * sizeof(Item), cudaMemcpyHostToDevice);
  return e != cudaSuccess ? e : cudaMemcpy(d_sched, start.data(), start.size() * sizeof(int), cudaMemcpyHostToDevice);
}

cudaError_t tc_configure(TcPlan* p, const TcConfig& c) {
  if (!tc_config_fits(p, c)) return cudaErrorInvalidValue;
  cudaError_t e;
  const int Bs = std::min(c.slice, p->B), nS = (p->B + Bs - 1) / Bs, NC = nc_of(Bs);
  const size_t xslice = (size_t)std::max(p->xtiles_inv, p->xtiles_fwd) * (p->bf16 ? 2 : 1) * NC * 128;
  if (xslice * nS != p->xbytes || !p->X) {
    if (p->X) {
      cudaFree(p->X);
      p->bytes -= p->xbytes;
      p->X = nullptr;
    }
    if ((e = tc_alloc((void**)&p->X, xslice * nS, &p->bytes)) != cudaSuccess) return e;
    p->xbytes = xslice * nS;
  }
  const size_t xsbytes = p->bf16 ? 0 : (xslice / 128 / 2) * nS * sizeof(float);  // a float a row pair
  if (xsbytes && (xsbytes != p->xsbytes || !p->XS)) {
    if (p->XS) {
      cudaFree(p->XS);
      p->bytes -= p->xsbytes;
      p->XS = nullptr;
    }
    if ((e = tc_alloc((void**)&p->XS, xsbytes, &p->bytes)) != cudaSuccess) return e;
    p->xsbytes = xsbytes;
  }
  // The rows of padding fields are the same in every tile of a slice, in both directions: zeroed here,
  // written by no call.  (Zeroed by every call, they were most of the tiles' writes with few fields: the
  // cached forward of one field at L = 128 took 59 us with split FP16 and 72 with split BF16, now 39 and 41.)
  if ((e = cudaMemset(p->X, 0, p->xbytes)) != cudaSuccess) return e;
  if (p->xsbytes && (e = cudaMemset(p->XS, 0, p->xsbytes)) != cudaSuccess) return e;
  if ((e = cudaDeviceSynchronize()) != cudaSuccess) return e;  // the calls' streams do not wait for the legacy one
  p->Bs = Bs;
  p->nS = nS;
  p->NC = NC;
  p->xslice = xslice;
  // Work order (the schedule then hands the items out in this order).  Grouped: the row blocks of
  // each group of 4 consecutive m run together, so that their data tiles are read from HBM about
  // once and the output rows of neighbouring m meet in L2.  Longest first: the classic order for
  // balance.  Order 0 (the default) is grouped in both directions.
  auto grouped = [](const Item& x, const Item& y) {
    if (x.m / 4 != y.m / 4) return x.m / 4 < y.m / 4;
    if (x.i != y.i) return x.i > y.i;
    return x.m < y.m;
  };
  auto longest_first = [](const Item& x, const Item& y) { return (x.c1 - x.c0) > (y.c1 - y.c0); };
  std::vector<Item> inv = p->inv_h, fwd = p->fwd_h;
  if (c.inv_order == 0) std::stable_sort(inv.begin(), inv.end(), grouped);
  else std::stable_sort(inv.begin(), inv.end(), longest_first);
  if (c.fwd_order == 0) std::stable_sort(fwd.begin(), fwd.end(), grouped);
  else std::stable_sort(fwd.begin(), fwd.end(), longest_first);
  if ((e = schedule(inv, p->grid_inv, p->items_inv, p->sched_inv)) != cudaSuccess) return e;
  if ((e = schedule(fwd, p->grid_fwd, p->items_fwd, p->sched_fwd)) != cudaSuccess) return e;
  p->smem = (size_t)c.stages * stage_bytes_of(NC, p->bf16) + 1024;
  p->cfg = c;
  return cudaSuccess;
}

TcConfig tc_config(const TcPlan* p) { return p->cfg; }

cudaError_t tc_setup(TcPlan** out, int L, int s, int B, int bf16, int device) {
  *out = nullptr;
  if (B < 1) return cudaErrorInvalidValue;
  TcPlan* p = new TcPlan();
  size_t ga = 0;
  p->bf16 = bf16 != 0;
  p->L = L;
  p->s = s;
  p->B = B;
  p->nC = (L + TK - 1) / TK;
  p->nI = (L + TM - 1) / TM;
  const int as = s < 0 ? -s : s;
  std::vector<Item>& inv = p->inv_h;
  std::vector<Item>& fwd = p->fwd_h;
  std::vector<long long> xoff(L), abase(L), ibase((size_t)L * std::max(1, (L + TM - 1) / TM), 0);
  std::vector<int> xc0(L);
  long long at = 0, ft = 0, xt = 0;
  for (int m = 0; m < L; ++m) {
    const int lmin = std::max(m, as), im = m / TM;
    xc0[m] = lmin / TK;
    xoff[m] = xt;
    xt += p->nC - xc0[m];
    abase[m] = ft;
    for (int i = im; i < p->nI; ++i) {
      // forward: rows l in block i with l >= m (rows l < |s| come out as zeros), K = m' <= l
      fwd.push_back({m, i, 0, std::min(p->nC, 4 * i + 4), ft});
      ft += 4 * i + 4;
    }
    for (int i = 0; i < p->nI; ++i) {
      // inverse: rows m' in block i, K = l >= max(m, m', |s|)
      const int c0 = std::max(lmin / TK, (i * TM) / TK);
      if (c0 < p->nC) {
        ibase[(size_t)m * p->nI + i] = at - c0;
        inv.push_back({m, i, c0, p->nC, at});
        at += p->nC - c0;
      }
    }
  }
  p->n_inv = (int)inv.size();
  p->n_fwd = (int)fwd.size();
  p->tiles_A = ft;
  p->tiles_inv = at;
  p->xtiles_inv = xt;
  p->xtiles_fwd = (long long)L * p->nC;
  cudaError_t e;
  {
    int sms = 0, optin = 0;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device)) != cudaSuccess) goto fail;
    if ((e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device)) != cudaSuccess) goto fail;
    p->grid = sms;
    p->smem_max = optin - 8192;  // the kernel's static shared memory and alignment slack
  }
  // the inverse leaves one SM to the recursion that writes the forward's operands meanwhile
  p->grid_inv = std::max(1, std::min(p->grid - 1, (int)inv.size()));
  p->grid_fwd = std::max(1, std::min(p->grid, (int)fwd.size()));
  if ((e = tc_alloc((void**)&p->items_inv, inv.size() * sizeof(Item), &p->bytes)) != cudaSuccess) goto fail;
  if ((e = tc_alloc((void**)&p->items_fwd, fwd.size() * sizeof(Item), &p->bytes)) != cudaSuccess) goto fail;
  if ((e = tc_alloc((void**)&p->sched_inv, (p->grid_inv + 1) * sizeof(int), &p->bytes)) != cudaSuccess) goto fail;
  if ((e = tc_alloc((void**)&p->sched_fwd, (p->grid_fwd + 1) * sizeof(int), &p->bytes)) != cudaSuccess) goto fail;
  ga = (size_t)(p->bf16 ? 2 : 1) * A_PART;  // bytes of an A tile in global memory
  if ((e = tc_alloc((void**)&p->A, (size_t)ft * ga, &p->bytes)) != cudaSuccess) goto fail;
  // zero once (entries no call writes stay zero); cudaMemset is asynchronous on the legacy
  // stream, and the plans' packing and recursions run on non-blocking streams: wait for it
  if ((e = cudaMemset(p->A, 0, (size_t)ft * ga)) != cudaSuccess) goto fail;
  if ((e = tc_alloc((void**)&p->A_inv, (size_t)at * ga, &p->bytes)) != cudaSuccess) goto fail;
  if ((e = cudaMemset(p->A_inv, 0, (size_t)at * ga)) != cudaSuccess) goto fail;
  if ((e = cudaDeviceSynchronize()) != cudaSuccess) goto fail;
  if ((e = tc_alloc((void**)&p->ibase, ibase.size() * sizeof(long long), &p->bytes)) != cudaSuccess) goto fail;
  if ((e = cudaMemcpy(p->ibase, ibase.data(), ibase.size() * sizeof(long long), cudaMemcpyHostToDevice)) != cudaSuccess)
    goto fail;
  if ((e = tc_alloc((void**)&p->abase, L * sizeof(long long), &p->bytes)) != cudaSuccess) goto fail;
  if ((e = tc_alloc((void**)&p->xoff, L * sizeof(long long), &p->bytes)) != cudaSuccess) goto fail;
  if ((e = tc_alloc((void**)&p->xc0, L * sizeof(int), &p->bytes)) != cudaSuccess) goto fail;
  if ((e = cudaMemcpy(p->abase, abase.data(), L * sizeof(long long), cudaMemcpyHostToDevice)) != cudaSuccess) goto fail;
  if ((e = cudaMemcpy(p->xoff, xoff.data(), L * sizeof(long long), cudaMemcpyHostToDevice)) != cudaSuccess) goto fail;
  if ((e = cudaMemcpy(p->xc0, xc0.data(), L * sizeof(int), cudaMemcpyHostToDevice)) != cudaSuccess) goto fail;
  {
    // Function attributes are process-wide upper bounds: the device's limit, so that plans of
    // every configuration can launch with their own amounts.
    if ((e = prefer_shared(pack_a_kernel<true, true>)) != cudaSuccess || (e = prefer_shared(pack_a_kernel<true, false>)) != cudaSuccess ||
        (e = prefer_shared(pack_a_kernel<false, true>)) != cudaSuccess || (e = prefer_shared(pack_a_kernel<false, false>)) != cudaSuccess)
      goto fail;
    if (p->bf16) {
      if ((e = gemm_attrs(tc_gemm_kernel<false, true>, p->smem_max)) != cudaSuccess) goto fail;
      if ((e = gemm_attrs(tc_gemm_kernel<true, true>, p->smem_max)) != cudaSuccess) goto fail;
      if ((e = prefer_shared(pack_v_kernel<true>)) != cudaSuccess) goto fail;
    } else {
      if ((e = gemm_attrs(tc_gemm_kernel<false, false>, p->smem_max)) != cudaSuccess) goto fail;
      if ((e = gemm_attrs(tc_gemm_kernel<true, false>, p->smem_max)) != cudaSuccess) goto fail;
      if ((e = prefer_shared(pack_v_kernel<false>)) != cudaSuccess) goto fail;
    }
  }
  {
    TcConfig c;  // as many stages as fit
    while (c.stages > 2 && !tc_config_fits(p, c)) --c.stages;
    if ((e = tc_configure(p, c)) != cudaSuccess) goto fail;
  }
  *out = p;
  return cudaSuccess;
fail:
  tc_destroy(p);
  return e;
}

void tc_destroy(TcPlan* p) {
  if (!p) return;
  void* ptrs[] = {p->items_inv, p->items_fwd, p->sched_inv, p->sched_fwd, p->A, p->A_inv, p->abase, p->ibase, p->X, p->XS, p->xoff, p->xc0};
  for (void* q : ptrs)
    if (q) cudaFree(q);
  delete p;
}

size_t tc_bytes(const TcPlan* p) { return p ? p->bytes : 0; }

InvTiles tc_inverse_tiles(const TcPlan* p) {
  InvTiles t;
  if (p) {
    t.A = p->A_inv;
    t.ibase = p->ibase;
    t.nI = p->nI;
    t.nC = p->nC;
    t.ntiles = p->tiles_inv;
    t.bf16 = p->bf16;
  }
  return t;
}

ATiles tc_a_tiles(const TcPlan* p) {
  ATiles t;
  if (p) {
    t.A = p->A;
    t.abase = p->abase;
    t.ntiles = p->tiles_A;
    t.bf16 = p->bf16;
  }
  return t;
}

cudaError_t tc_pack_a(TcPlan* p, int forward, const double* table, const float* U, cudaStream_t st, int* launches) {
  // one block per (item, chunk): grid.x covers the longest item (at most nC chunks), grid.y the items
  const dim3 gf(p->nC, p->n_fwd), gi(p->nC, p->n_inv);
  if (forward && p->bf16)
    pack_a_kernel<true, true><<<gf, 256, 0, st>>>(p->L, p->s, p->items_fwd, table, U, p->A, p->tiles_A);
  else if (forward)
    pack_a_kernel<true, false><<<gf, 256, 0, st>>>(p->L, p->s, p->items_fwd, table, U, p->A, p->tiles_A);
  else if (p->bf16)
    pack_a_kernel<false, true><<<gi, 256, 0, st>>>(p->L, p->s, p->items_inv, table, U, p->A_inv, p->tiles_inv);
  else
    pack_a_kernel<false, false><<<gi, 256, 0, st>>>(p->L, p->s, p->items_inv, table, U, p->A_inv, p->tiles_inv);
  *launches += 1;
  return cudaGetLastError();
}

cudaError_t tc_pack_data(TcPlan* p, const void* src, cudaStream_t st, int* launches) {
  // Two fields a CTA while eight would give fewer than two CTAs to an SM (L = 65, B = 8, kept Delta, inverse: split BF16 49.7 -> 39.7 us)
  const int mb = (p->L + 15) / 16, per = p->nC * mb * p->nS * ((p->Bs + 7) / 8) < 2 * p->grid ? 2 : 8;
  const dim3 g(p->nC, mb, (unsigned)(p->nS * ((p->Bs + per - 1) / per)));
  if (p->bf16)
    pack_v_kernel<true><<<g, 256, 0, st>>>(p->L, p->s, p->B, p->Bs, per, p->xslice, p->NC, p->xc0, p->xoff,
                                           (const float2*)src, p->X, p->XS);
  else
    pack_v_kernel<false><<<g, 256, 0, st>>>(p->L, p->s, p->B, p->Bs, per, p->xslice, p->NC, p->xc0, p->xoff,
                                            (const float2*)src, p->X, p->XS);
  *launches += 1;
  return cudaGetLastError();
}

TileOut tc_forward_tiles(const TcPlan* p) {
  TileOut o;
  o.X = p->X;
  o.NC = p->NC;
  o.nC = p->nC;
  o.mode = p->bf16 ? 2 : 1;
  o.Bs = p->Bs;
  o.xslice = p->xslice;
  o.xbytes = p->xbytes;
  o.scale = p->XS;
  return o;
}

// The forward's rows l of one order lie 2l apart in flm: written from the GEMM, every 8-byte value is a
// sector of its own, which meets its neighbours' (other orders, other CTAs) in L2 only while the output
// is small.  From 2^22 coefficients (32 MB) on, the GEMM writes half rows, contiguous in l, into the
// workspace and rows_to_flm_kernel transposes them (GB300, B = 64: the GEMM at L = 1024 1.68 ms direct, 0.69 by rows and 0.17 for the transposition).
constexpr long long kRowsFrom = 1ll << 22;

cudaError_t tc_gemm(TcPlan* p, int forward, void* out, void* rows, int* status, long long wait_ns,
                    cudaStream_t st, int* launches) {
  const bool via_rows = forward && rows && (long long)p->B * p->L * p->L >= kRowsFrom;
  // all slices of fields in one launch, one after the other; every slice reads the same A tiles (a launch a slice took
  // 8 to 10 us each at small band-limits: split BF16, L = 8, B = 8192 2607 us an inverse and a forward, now 173; tf32x3, L = 33,
  // B = 8192 3661, now 1513)
  TcArgs a;
  a.L = p->L;
  a.s = p->s;
  a.B = p->B;
  a.Bs = p->Bs;
  a.NC = p->NC;
  a.stages = p->cfg.stages;
  a.sched = forward ? p->sched_fwd : p->sched_inv;
  a.items = forward ? p->items_fwd : p->items_inv;
  a.A = forward ? p->A : p->A_inv;
  a.X = p->X;
  a.xslice = p->xslice;
  a.XS = p->XS;
  a.xoff = p->xoff;
  a.xc0 = p->xc0;
  a.out = (float2*)(via_rows ? rows : out);
  a.rows = via_rows;
  a.status = status;
  a.wait_ns = wait_ns;
  a.a_tiles = forward ? p->tiles_A : p->tiles_inv;
  a.x_tiles = (long long)(p->xslice / ((p->bf16 ? 2 : 1) * (size_t)p->NC * 128));
  a.out_field = (long long)((forward && !via_rows) ? p->L : 2 * p->L - 1) * p->L;
  const dim3 grid((unsigned)(forward ? p->grid_fwd : p->grid_inv), (unsigned)p->nS);
  if (forward && p->bf16)
    tc_gemm_kernel<true, true><<<grid, THREADS, p->smem, st>>>(a);
  else if (forward)
    tc_gemm_kernel<true, false><<<grid, THREADS, p->smem, st>>>(a);
  else if (p->bf16)
    tc_gemm_kernel<false, true><<<grid, THREADS, p->smem, st>>>(a);
  else
    tc_gemm_kernel<false, false><<<grid, THREADS, p->smem, st>>>(a);
  *launches += 1;
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (via_rows) {
    const int N = 2 * p->L - 1;
    // fields in z, at most 65535 a launch (the library's largest batch)
    rows_to_flm_kernel<<<dim3((p->L + 31) / 32, (N + 31) / 32, p->B), 256, 0, st>>>(
        p->L, (const float2*)rows, (float2*)out, (long long)p->B * N * p->L, (long long)p->B * p->L * p->L);
    *launches += 1;
    return cudaGetLastError();
  }
  return cudaSuccess;
}

SSHT_BOUNDS_TU(contract_tc)

}  // namespace ssht
