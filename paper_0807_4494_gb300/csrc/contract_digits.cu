// The contractions of FP64 plans (contract_simt.cu gives the formulas) on the tensor cores, both operands in
// fixed-point digits held as FP16 (digits.cuh; torus_digits.cu says why the sums are exact).
//
// For an order m the inverse is F_{+-m}[m'] = sum_l A[m', l] sf_{l,+-m}, the projection sf_{l,+-m} = sum_m' A[m', l] H_{+-m}[m'], with
// A[m', l] = U_l[m'] Delta^l_{m' m} up to signs.  A work item is 128 rows (m' or l) of one order and four or eight fields: 16 or 32
// columns (field, sign of m, part).  A CTA makes the digits of A itself, from the FP64 table into the tensor cores' shared memory: 16
// warps, a thread one row and eight k's at a time.  A's entries have one power of two for all of them (|A| <= sqrt((2L - 1) / 4 pi))
// and nine digits, so that they keep 2^-58 of that bound; a data column has its own and eight.  44 products of digits a chunk.
//
// What bounds it: making A's digits, 6000 clocks a chunk of 4096 entries -- loads, one FP64 product an entry (2048 clocks; CUDA
// cores need four more a field) and the integer instructions behind it, with 60 % of the issue slots busy; the
// tensor cores' part (1440) is beside it.  L = 512, B = 1: 270 us the inverse and 288 the projection, 517 and 482 on CUDA
// cores; L = 256, B = 8 176 both (245 in two items of four fields), 881 there.  The next chunk's FP64 products stand one by one among the integer
// instructions (281 and 286 us before).  Taken back: the conversion to integers by F2I (307 and 333 us: it runs at the FP64 pipe's
// rate), fewer instructions to take the digits out (280 and 299: within the noise).
#include <algorithm>
#include <cmath>
#include <cstdint>

#include "bounds.cuh"
#include "digits.cuh"
#include "ssht_internal.h"

namespace ssht {
namespace {

constexpr int kADigits = 9, kStages = 2;
constexpr int kAPart = 128 * 128, kATile9 = (kADigits + 1) / 2 * kAPart;  // a part: two digits' 32 k's
// Fields of a work item: four or eight.
template <int FIELDS> constexpr int kCols = 4 * FIELDS;
template <int FIELDS> constexpr int kXPart = kCols<FIELDS> * 128;
template <int FIELDS> constexpr int kXTile = kDigits / 2 * kXPart<FIELDS>;
template <int FIELDS> constexpr int kStageBytes = kATile9 + kXTile<FIELDS>;
template <int FIELDS> constexpr size_t kSmem = (size_t)kStages * kStageBytes<FIELDS> + 1024;
constexpr int kGenWarps = 16, kThreads = 128 + 32 * kGenWarps;
constexpr int kRegsIssue = 32, kRegsGen = 112;                    // 128 * 32 + 512 * 112 = 640 * 96
constexpr int kMaxL = 512;                                        // an item's sums are one segment of at most 512 k's

// Offsets of degree l in U and in the table: below 2^31 up to kMaxL.
__device__ __forceinline__ int tri32(int m) { return m * (m + 1) / 2; }
__device__ __forceinline__ int doff32(int l) { return l * (l + 1) * (2 * l + 1) / 6; }
__host__ __device__ inline int chunks_of(int L) { return (L + 31) / 32; }

// (-1)^{s + e} i^k (x, y): parts exchanged and signs flipped, no arithmetic
__device__ __forceinline__ double2 times_ik(int s, int e, int k, double x, double y) {
  const int r = ((k + 2 * (s + e)) % 4 + 4) % 4;
  return make_double2(r == 0 ? x : r == 1 ? -y : r == 2 ? -x : y, r == 0 ? y : r == 1 ? x : r == 2 ? -y : -x);
}

// ---------------------------------------------------------------------------------------------
// Data columns: tiles [m][field / FIELDS][chunk] of 4 FIELDS rows
// ---------------------------------------------------------------------------------------------
// A CTA takes kSources (field, order |m|), each two complex columns -- four rows -- of all k: their largest
// exponents, then their digits.  The lanes run along orders (inverse: sf_{l,+-m}, contiguous in m) or k (projection: H).
constexpr int kSources = 2, kPackThreads = 128;

struct PackArgs {
  int L, s, B, groups;
  const double2* in;
  long long in_n;
  uint8_t* x;
  int* exps;
  long long x_n, exps_n;  // tiles and exponents of the workspace
};

template <bool FWD, int FIELDS>
__global__ void __launch_bounds__(kPackThreads) digit_columns_kernel(const __grid_constant__ PackArgs a) {
  __shared__ int top[kSources][4];
  const int L = a.L, nc = chunks_of(L), pieces = 4 * nc, items = kSources * pieces, as = a.s < 0 ? -a.s : a.s;
  if (threadIdx.x < kSources * 4) top[threadIdx.x >> 2][threadIdx.x & 3] = 1;
  __syncthreads();
  double x[4][8];
  auto load = [&](int b, int m, int g) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int k = FWD ? 32 * (g >> 2) + 4 * i + (g & 3) : 8 * g + i;
      double2 u = make_double2(0.0, 0.0), v = u;
      if (FWD) {
        if (k < L) {  // H_{+-m}[m' = k], (-1)^{m'} for +m
          const long long o = ((long long)b * (2 * L - 1) + L - 1 + m) * L + k, on = o - 2ll * m * L;
          if (in_bounds(o, a.in_n, kbSimtIn)) u = __ldg(&a.in[o]);
          if (m > 0 && in_bounds(on, a.in_n, kbSimtIn)) v = __ldg(&a.in[on]);
          if (k & 1) u = make_double2(-u.x, -u.y);
        }
      } else if (k < L && k >= m && k >= as) {  // sf_{l = k, +-m}, (-1)^l for -m
        const long long o = (long long)b * L * L + (long long)k * k + k + m, on = o - 2 * m;
        if (in_bounds(o, a.in_n, kbSimtIn)) u = __ldg(&a.in[o]);
        if (m > 0 && in_bounds(on, a.in_n, kbSimtIn)) v = __ldg(&a.in[on]);
        if (i & 1) v = make_double2(-v.x, -v.y);
      }
      x[0][i] = u.x;
      x[1][i] = u.y;
      x[2][i] = v.x;
      x[3][i] = v.y;
    }
  };
#pragma unroll 1
  for (int phase = 0; phase < 2; ++phase) {
#pragma unroll 1
    for (int w = threadIdx.x; w < items; w += kPackThreads) {
      const int so = FWD ? w / pieces : w % kSources, g = FWD ? w - so * pieces : w / kSources;
      const long long src = (long long)blockIdx.x * kSources + so;
      if (src >= (long long)a.B * L) continue;
      const int b = (int)(src / L), m = (int)(src - (long long)b * L);
      if (!FWD && (g >> 2) < m / 32) continue;  // below the order: no item reads it
      if (phase == 0 || items > kPackThreads) load(b, m, g);  // else its values are still here
      const size_t tile = (size_t)m * a.groups + b / FIELDS;
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        if (phase == 0) {
          int e = 1;
#pragma unroll
          for (int k = 0; k < 8; ++k) e = max(e, exponent_of(x[r][k]));
          if (e > *(volatile int*)&top[so][r]) atomicMax(&top[so][r], e);
        } else {
          const int row = 4 * (b % FIELDS) + r, e = top[so][r];
          const long long ei = (long long)tile * kCols<FIELDS> + row, xi = (long long)tile * nc + (g >> 2);
          if ((g >> 2) == nc - 1 && (g & 3) == 0 && in_bounds(ei, a.exps_n, kbDigitExp)) a.exps[ei] = e;
          if (in_bounds(xi, a.x_n, kbDigitTile)) put_digits<kDigits, kXPart<FIELDS>>(a.x + (size_t)xi * kXTile<FIELDS>, row, g & 3, x[r], e);
        }
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------------------------
// Products
// ---------------------------------------------------------------------------------------------
struct GemmArgs {
  int L, s, B, groups, mblocks, nitems, aexp;  // aexp: exponent field of A's power of two
  const double* table;
  const double* U;
  const uint8_t* x;
  const int* xexp;
  long long x_n, exps_n;  // tiles and exponents of the workspace
  double2* out;
  long long out_n;
  int* status;
  long long wait_ns;
};

// Work item w: order m, row block i, fields FIELDS g on, chunks c0 .. c1 - 1 (none: nothing to do).  The row
// blocks with the longest sums come first, so that every CTA gets its share of each.
struct Item {
  int m, i, g, c0, c1;
};
template <bool FWD>
__device__ __forceinline__ Item item_of(const GemmArgs& a, int w) {
  Item t;
  t.g = w % a.groups;
  const int r = w / a.groups;
  t.i = r / a.L;
  t.m = r - t.i * a.L;
  if (FWD) {
    t.i = a.mblocks - 1 - t.i;
    t.c0 = 0;
    t.c1 = t.m >= 128 * (t.i + 1) ? 0 : chunks_of(min(128 * (t.i + 1), a.L));
  } else {
    t.c0 = max(max(t.m, 128 * t.i), a.s < 0 ? -a.s : a.s) / 32;
    t.c1 = chunks_of(a.L);
  }
  return t;
}

// Column of accumulator d: the even ones, then the odd ones.
template <int FIELDS>
__device__ __forceinline__ constexpr uint32_t acc_col(int d) { return kCols<FIELDS> * (d >> 1) + (d & 1) * 5 * kCols<FIELDS>; }

template <bool FWD, int FIELDS>
__global__ void __launch_bounds__(kThreads, 1) digit_contract_kernel(const __grid_constant__ GemmArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t full[kStages], data_full[kStages], empty[kStages], acc_full[2], acc_empty[2], done_bar;
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag;
  constexpr int COLS = kCols<FIELDS>, STAGE = kStageBytes<FIELDS>, XTILE = kXTile<FIELDS>, XPART = kXPart<FIELDS>;
  constexpr bool kTwo = FIELDS == 4;  // two sets of accumulators fit the tensor memory
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp == 1) tmem_alloc(&tmem_base, 512);
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], kGenWarps);
      mbar_init(&data_full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int k = 0; k < 2; ++k) {
      mbar_init(&acc_full[k], 1);
      mbar_init(&acc_empty[k], kGenWarps);
    }
    mbar_init(&done_bar, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tbase = tmem_base;
  volatile int* abort = &abort_flag;
  const int L = a.L, nc = chunks_of(L);

  if (warp < 4) {
    regs_dec<kRegsIssue>();
    if (warp == 0) {
      // ---- the data tiles ----
      const bool one = elect_one();
      int s = 0, ph = 1;
      uint32_t used = 0, uph = 0;  // stages that were filled, and the parity of their last fill
      for (int w = blockIdx.x; w < a.nitems && going(abort); w += gridDim.x) {
        const Item t = item_of<FWD>(a, w);
        const long long x0 = ((long long)t.m * a.groups + t.g) * nc;
        for (int c = t.c0; c < t.c1; ++c) {
          if (!__all_sync(0xffffffffu, mbar_wait(&empty[s], ph, abort, a.wait_ns))) {
            *abort = 1;
            break;
          }
          if (one) {
            mbar_expect_tx(&data_full[s], (uint32_t)XTILE);
            // (a tile outside the workspace is recorded and tile 0 copied instead: the pipeline still completes)
            const long long xi = in_bounds(x0 + c, a.x_n, kbDigitTile) ? x0 + c : 0;
            bulk_g2s(smem + s * STAGE + kATile9, a.x + (size_t)xi * XTILE, XTILE, &data_full[s]);
          }
          used |= 1u << s;
          uph = (uph & ~(1u << s)) | ((uint32_t)(ph ^ 1) << s);
          if (++s == kStages) {
            s = 0;
            ph ^= 1;
          }
        }
      }
      // every issued copy must have landed before the CTA leaves
      for (int k = 0; k < kStages; ++k)
        if ((used >> k) & 1u) mbar_wait(&data_full[k], (uph >> k) & 1u, nullptr, kDrainNs);
    } else if (warp == 1) {
      // ---- MMA issuer: digits i of A and j of the data into accumulator i + j <= 8.  A part of the data tile
      // holds two digits, so the even (or the odd) ones are the rows of one operand, and with the accumulators of one
      // parity side by side one product takes digit i times all of them ----
      const bool one = elect_one();
      const uint32_t lo0 = (smem_u32(smem) >> 4) + kDescLow;
      int s = 0, ph = 0, buf = 0, bph = 1;
      for (int w = blockIdx.x; w < a.nitems && going(abort); w += gridDim.x) {
        const Item t = item_of<FWD>(a, w);
        if (t.c1 <= t.c0) continue;
        for (int c = t.c0; c < t.c1; ++c) {
          const bool here = (c > t.c0 || mbar_wait(&acc_empty[buf], bph, abort, a.wait_ns)) && mbar_wait(&full[s], ph, abort, a.wait_ns) &&
                            mbar_wait(&data_full[s], ph, abort, a.wait_ns);
          if (!__all_sync(0xffffffffu, here)) {
            *abort = 1;
            break;
          }
          fence_after();
          if (one) {
            const uint32_t la = lo0 + (uint32_t)(s * (STAGE >> 4)), lb = la + (kATile9 >> 4), dt = tbase + 256u * buf;
            const uint32_t more = c > t.c0 ? 1u : 0u;
#pragma unroll
            for (int kk = 0; kk < 2; ++kk)
#pragma unroll
              for (int i = 0; i < kADigits; ++i) {
                const int jm = kDigits - 1 < kADigits - 1 - i ? kDigits - 1 : kADigits - 1 - i, even = jm / 2 + 1, odd = (jm + 1) / 2;
                const uint32_t da = la + (i >> 1) * (kAPart >> 4) + (i & 1) * 4 + 2 * kk, init = kk == 0 && i == 0 ? more : 1u;
                mma_f16_lo<false>(dt + acc_col<FIELDS>(i), da, lb + 2 * kk, idesc_f16(128, COLS * even), init);
                if (i == 1) {  // accumulator 8 has its first product here
                  mma_f16_lo<false>(dt + acc_col<FIELDS>(2), da, lb + 4 + 2 * kk, idesc_f16(128, COLS * (odd - 1)), 1u);
                  mma_f16_lo<false>(dt + acc_col<FIELDS>(8), da, lb + (odd - 1) * (XPART >> 4) + 4 + 2 * kk, idesc_f16(128, COLS), kk == 0 ? more : 1u);
                } else if (odd) {
                  mma_f16_lo<false>(dt + acc_col<FIELDS>(i + 1), da, lb + 4 + 2 * kk, idesc_f16(128, COLS * odd), init);
                }
              }
            mma_commit(&empty[s]);
            if (c + 1 == t.c1) mma_commit(&acc_full[buf]);
          }
          __syncwarp();
          if (++s == kStages) {
            s = 0;
            ph ^= 1;
          }
        }
        if (kTwo) buf ^= 1;
        if (buf == 0) bph ^= 1;
      }
      // every issued product has completed before the CTA leaves
      if (one) mma_commit(&done_bar);
      __syncwarp();
      mbar_wait(&done_bar, 0, nullptr, kDrainNs);
    }
  } else {
    // ---- A's digits; the accumulators of an item once two chunks of the next are under way ----
    regs_inc<kRegsGen>();
    const int gt = threadIdx.x - 128, as = a.s < 0 ? -a.s : a.s;
    // a thread's row and piece of eight k's: lanes along the table's contiguous m'
    const int row = FWD ? gt >> 2 : gt & 127, piece = FWD ? gt & 3 : gt >> 7;
    const int q = warp & 3, cg = (warp - 4) >> 2;
    const uint32_t tq = tbase + ((uint32_t)(q * 32) << 16) + FIELDS * cg;
    int s = 0, ph = 1, buf = 0, bph = 0;

    auto drain = [&](const Item& t) {  // false: gave up
      if (!__all_sync(0xffffffffu, mbar_wait(&acc_full[buf], bph, abort, a.wait_ns))) {
        *abort = 1;
        return false;
      }
      fence_after();
      const uint32_t acc = tq + 256 * buf;
      const int r = 128 * t.i + 32 * q + lane, m = t.m;
#pragma unroll
      for (int f = 0; f < FIELDS / 4; ++f) {
        uint32_t v[kADigits][4];
        __syncwarp();
#pragma unroll
        for (int d = 0; d < kADigits; ++d) tmem_ld4_nowait(acc + acc_col<FIELDS>(d) + 4 * f, v[d]);
        tmem_wait_ld();
        if (f + 1 == FIELDS / 4) {  // all is read
          fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&acc_empty[buf]);
          if (kTwo) buf ^= 1;
          if (buf == 0) bph ^= 1;
        }
        const int b = FIELDS * t.g + cg * (FIELDS / 4) + f;
        if (b >= a.B || r >= L || (FWD && r < m)) continue;
        const long long ei = ((long long)m * a.groups + t.g) * COLS + FIELDS * cg + 4 * f;
        if (!in_bounds(ei + 3, a.exps_n, kbDigitExp)) continue;
        const int4 e = __ldg((const int4*)(a.xexp + ei));
        const int xe[4] = {e.x, e.y, e.z, e.w};
        double z[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          int d[kADigits];  // whole numbers of at most min(i + 1, 8) 2^21
#pragma unroll
          for (int i = 0; i < kADigits; ++i) d[i] = __float2int_rn(__uint_as_float(v[i][k]));
          const long long hi = (long long)(d[0] * 128 + d[1]) * 16384 + (d[2] * 128 + d[3]);
          const long long lo = ((long long)(d[4] * 128 + d[5]) * 16384 + (d[6] * 128 + d[7])) * 128 + d[8];
          z[k] = assemble(hi * 128, lo, a.aexp + xe[k] - 2112);
        }
        if (FWD) {  // +m: (-1)^m; -m: (-1)^{l+m}
          const long long o = (long long)b * L * L + (long long)r * r + r + m;
          if (in_bounds(o, a.out_n, kbSimtOut)) a.out[o] = times_ik(a.s, m, m + a.s, z[0], z[1]);
          if (m > 0 && in_bounds(o - 2 * m, a.out_n, kbSimtOut)) a.out[o - 2 * m] = times_ik(a.s, r + m, a.s - m, z[2], z[3]);
        } else {  // +m: (-1)^{m'-m}; -m: (-1)^m
          const long long o = ((long long)b * (2 * L - 1) + L - 1 + m) * L + r, on = o - 2ll * m * L;
          if (in_bounds(o, a.out_n, kbSimtOut)) a.out[o] = times_ik(a.s, r - m, -(m + a.s), z[0], z[1]);
          if (m > 0 && in_bounds(on, a.out_n, kbSimtOut)) a.out[on] = times_ik(a.s, m, m - a.s, z[2], z[3]);
        }
      }
      return true;
    };

    // Delta and U of eight k's of a chunk (masked ones from a valid place)
    double d[8], u[8];
    auto fetch = [&](const Item& t, int c) {
      const int r = 128 * t.i + row;
      if (FWD) {  // row l = r; k = 4 i + piece of the chunk (the columns are packed alike): four lanes read 32 bytes
        const int k0 = 32 * c + piece, last = r < L && r >= t.m && r >= as ? r : -1;
        const int o = last < 0 ? 0 : doff32(r) + t.m * (r + 1), ou = last < 0 ? 0 : tri32(r);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int mp = k0 + 4 * i <= last ? k0 + 4 * i : 0;
          const bool here = in_bounds(o + mp, doff32(L), kbDigitTable) && in_bounds(ou + mp, tri32(L), kbDigitTable);
          d[i] = __ldg(&a.table[here ? o + mp : 0]);
          u[i] = __ldg(&a.U[here ? ou + mp : 0]);
          if (k0 + 4 * i > last) u[i] = 0.0;
        }
      } else {  // row m' = r; k = l
        const int l0 = 32 * c + 8 * piece, from = r < L ? max(max(r, t.m), as) : L;
        int o = doff32(l0) + t.m * (l0 + 1) + r, ou = tri32(l0) + r;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const bool in = l0 + i >= from && l0 + i < L && in_bounds(o, doff32(L), kbDigitTable) && in_bounds(ou, tri32(L), kbDigitTable);
          d[i] = __ldg(&a.table[in ? o : 0]);
          u[i] = __ldg(&a.U[in ? ou : 0]);
          if (!in) u[i] = 0.0;
          o += (l0 + i + 1) * (l0 + i + 1) + t.m;
          ou += l0 + i + 1;
        }
      }
    };
    auto next_item = [&](int& w, Item& t) {  // the next one with something to do
      while (w < a.nitems) {
        t = item_of<FWD>(a, w);
        if (t.c1 > t.c0) return true;
        w += gridDim.x;
      }
      return false;
    };
    // where the loads are: one chunk ahead of the products U Delta, two ahead of the digits
    Item ft;
    int fw = blockIdx.x, fc = 0;
    bool loads = next_item(fw, ft);
    auto next_loads = [&] {
      if (loads && ++fc >= ft.c1) {
        fw += gridDim.x;
        loads = next_item(fw, ft);
        fc = ft.c0;
      }
      if (loads) fetch(ft, fc);
    };
    Item pending, t = ft;
    pending.m = -1;
    int w = fw;
    bool more = loads;
    double x[8];
    if (more) {
      fc = ft.c0;
      fetch(ft, fc);
#pragma unroll
      for (int i = 0; i < 8; ++i) x[i] = u[i] * d[i];
      next_loads();
    }
    while (more && going(abort)) {
      bool ok = true;
      for (int c = t.c0; c < t.c1; ++c) {
        // the next chunk's products, one by one among the integer instructions: the FP64 pipe holds a warp for 64 clocks
        unsigned long long v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          v[i] = (unsigned long long)fixed_point<7 * kADigits - 54>(x[i], a.aexp);
          x[i] = u[i] * d[i];
        }
        next_loads();
        if (!__all_sync(0xffffffffu, mbar_wait(&empty[s], ph, abort, a.wait_ns))) {
          *abort = 1;
          ok = false;
          break;
        }
        put_integers<kADigits, kAPart>(smem + s * STAGE, row, piece, v);
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) mbar_arrive(&full[s]);
        if (++s == kStages) {
          s = 0;
          ph ^= 1;
        }
        if (pending.m >= 0 && (c == t.c0 + 1 || c + 1 == t.c1)) {
          ok = drain(pending);
          __syncwarp();
          pending.m = -1;
          if (!ok) break;
        }
      }
      if (!ok) break;
      pending = t;
      w += gridDim.x;
      more = next_item(w, t);
    }
    __syncwarp();
    if (pending.m >= 0 && going(abort)) drain(pending);
  }
  fence_before();
  __syncthreads();
  fence_after();
  if (*abort && threadIdx.x == 0) atomicOr(a.status, 2);
  if (warp == 1) tmem_dealloc(tbase, 512);
}

// Four fields an item (two sets of accumulators then fit the tensor memory), or eight beyond that: A's digits, the larger
// part of the work, are made once for them (L = 256, B = 8 245 -> 176 us, L = 64, B = 64 151 -> 127).
int fields_of(int B) { return B > 4 ? 8 : 4; }
int groups_of(int B) { return (B + fields_of(B) - 1) / fields_of(B); }

template <bool FWD, int FIELDS>
cudaError_t run(int L, int s, int B, int sms, const double* table, const double* U, const void* in, size_t in_bytes, void* work,
                size_t work_bytes, void* out, size_t out_bytes, int* status, long long wait_ns, cudaStream_t st) {
  PackArgs k{};
  k.L = L;
  k.s = s;
  k.B = B;
  k.groups = groups_of(B);
  k.in = (const double2*)in;
  k.in_n = (long long)(in_bytes / sizeof(double2));
  k.x = (uint8_t*)work;
  k.x_n = (long long)L * k.groups * chunks_of(L);
  k.exps_n = (long long)L * k.groups * kCols<FIELDS>;
  k.exps = (int*)((uint8_t*)work + (size_t)k.x_n * kXTile<FIELDS>);
  if ((size_t)k.x_n * kXTile<FIELDS> + (size_t)k.exps_n * sizeof(int) > work_bytes) return cudaErrorInvalidValue;
  digit_columns_kernel<FWD, FIELDS><<<(unsigned)(((long long)B * L + kSources - 1) / kSources), kPackThreads, 0, st>>>(k);
  GemmArgs a{};
  a.L = L;
  a.s = s;
  a.B = B;
  a.groups = k.groups;
  a.mblocks = (L + 127) / 128;
  a.nitems = L * a.mblocks * a.groups;
  // |U Delta| <= sqrt((2L - 1) / 4 pi) < 2^e, and A's integers below 2^62 of the field e + 1022
  int e = 0;
  std::frexp(std::sqrt((2.0 * L - 1) / 12.566370614359172), &e);
  a.aexp = 1022 + std::max(e, 0);
  a.table = table;
  a.U = U;
  a.x = k.x;
  a.xexp = k.exps;
  a.x_n = k.x_n;
  a.exps_n = k.exps_n;
  a.out = (double2*)out;
  a.out_n = (long long)(out_bytes / sizeof(double2));
  a.status = status;
  a.wait_ns = wait_ns;
  digit_contract_kernel<FWD, FIELDS><<<(unsigned)std::min(a.nitems, sms), kThreads, kSmem<FIELDS>, st>>>(a);
  return cudaGetLastError();
}

}  // namespace

// Where they beat the CUDA cores' contractions, an inverse and a projection in us, these and those: L = 512, B = 1 594 and 1006,
// B = 4 627 and 3041; L = 256, B = 1 136 and 168, B = 8 176 and 881; L = 192, B = 8 133 and 413; L = 129, B = 4 75 and 92; L = 64,
// B = 64 127 and 208.  Below B L^3 = 2^23 few items, of few chunks, leave the launch and the epilogue (L = 192, B = 1 109 and 98;
// L = 160, B = 1 86 and 63), and below L = 64 half of a tile's rows are empty (L = 40, B = 96 156 and 126).
bool contract_digits_wanted(int L, int B) { return L >= 64 && L <= kMaxL && (long long)B * L * L * L > (1ll << 23); }

size_t contract_digits_bytes(int L, int B) {
  const size_t cols = 4 * fields_of(B);
  return (size_t)L * groups_of(B) * cols * (chunks_of(L) * (size_t)(kDigits * 64) + sizeof(int));
}

template <bool FWD, int FIELDS>
static cudaError_t kernel_attr() {
  cudaError_t e = prefer_shared(digit_contract_kernel<FWD, FIELDS>);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(digit_contract_kernel<FWD, FIELDS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem<FIELDS>);
}

cudaError_t contract_digits_setup() {
  cudaError_t e = kernel_attr<false, 4>();
  if (e == cudaSuccess) e = kernel_attr<true, 4>();
  if (e == cudaSuccess) e = kernel_attr<false, 8>();
  if (e == cudaSuccess) e = kernel_attr<true, 8>();
  return e;
}

cudaError_t contract_digits(int forward, int L, int s, int B, int sms, const double* table, const double* U, const void* in,
                            size_t in_bytes, void* work, size_t work_bytes, void* out, size_t out_bytes, int* status,
                            long long wait_ns, cudaStream_t st) {
  auto go = fields_of(B) == 8 ? (forward ? run<true, 8> : run<false, 8>) : (forward ? run<true, 4> : run<false, 4>);
  return go(L, s, B, sms, table, U, in, in_bytes, work, work_bytes, out, out_bytes, status, wait_ns, st);
}

SSHT_BOUNDS_TU(contract_digits)

}  // namespace ssht
