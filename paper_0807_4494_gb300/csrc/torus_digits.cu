// Torus passes of FP64 plans on the tensor cores: the folded cosine and sine products of the torus stage
// (torus_gemm.cu gives the identities) with both operands in fixed point, eight signed digits of seven bits held
// as FP16 (Ozaki, Ogita, Oishi, Rump, "Error-free transformations of matrix multiplication", Numer. Algorithms
// 59, 2012).
//
// A row of an operand -- a matrix row, or the real or imaginary part of a data column, over all k -- is
// scaled by one power of two to 55-bit integers x = sum_i d_i 128^(7-i), -64 <= d_i <= 64.  Products of digits i
// and j with i + j = d add up in the tensor memory's accumulator d: whole numbers of at most
// 2^12 * 8 * 512 = 2^24 in a segment of 512 k, so FP32 adds them without rounding.  The 36 products with i + j <= 7 are
// taken; what is left out is below 2^-57 of the rows' largest products.  The accumulators are put together as
// 64-bit integers and rounded once to FP64.  The transforms' error is what it was with FFTs (round trip against
// exact sums 2.3e-13 at L = 512, 2.8e-14 at L = 129, with both).
//
// What bounds it: the tensor cores (36 digit products of 128 x 64 x 16 in 15 instructions, 1150 clocks, and 132 KB of operands
// read from shared memory, 1060), and below L = 300 launches, the first loads and the epilogue (10 us a pass).  It replaces FFTs of odd
// length and the kernels between them, which the FP64 pipe bounds: that pipe does two multiply-adds a clock on
// an SM.  Torus stage of an inverse and a forward, before and now: L = 512, B = 1 1003 and 200 us (a product 35 us, 43 with
// an instruction for each pair of digits; a packing 12); L = 129, B = 4 587 and 105; L = 256, B = 8 2088 and 245.
// The tile is 128 rows x 32 complex columns: eight accumulators of 64 columns fill the tensor memory.
#include <algorithm>
#include <cstdint>

#include "bounds.cuh"
#include "digits.cuh"
#include "ssht_internal.h"
#include "torus_matrices.cuh"

namespace ssht {
namespace {

constexpr int kChunkK = 32;                                  // k's of a tile
constexpr int kMatTile = 128 * kChunkK * kDigits * 2;        // four parts of 128 rows x 128 bytes: two digits' 32 k's
template <int PAIRS> constexpr int kDataTile = 2 * PAIRS * kChunkK * kDigits * 2;  // PAIRS complex columns
template <int PAIRS> constexpr int kStageBytes = kMatTile + kDataTile<PAIRS>;
constexpr int kStages = 2;
constexpr int kSegChunks = 16;                               // chunks whose sums stay exact: 512 k
constexpr int kEpiWarps = 16, kThreads = 128 + 32 * kEpiWarps;
constexpr int kRegsIssue = 32, kRegsEpilogue = 112;          // 128 * 32 + 512 * 112 = 640 * 96
template <int PAIRS> constexpr size_t kSmem = (size_t)kStages * kStageBytes<PAIRS> + 1024;

enum Pass { kThetaInverse = 0, kPhiInverse, kPhiForward, kThetaForward, kThetaAdjoint };
enum Matrix { kCosKX = 0, kSinKX, kCosXK, kSinXK, kWeightE, kWeightO, kMatrices };

// The columns of a pass come in two sets, each with its matrix: the orders |m| of each parity of m + s
// (cosines for the even ones) in the theta passes, cosines and sines of a ring in the phi passes.
struct Sets {
  int n[2];      // complex columns
  int tiles[2];  // data tiles
  __host__ __device__ int all() const { return tiles[0] + tiles[1]; }
};

__host__ __device__ inline bool by_order(int pass) { return pass == kThetaInverse || pass >= kThetaForward; }
// |m| of a parity class: first, first + 2, ...
__host__ __device__ inline int first_order(int cls, int s) { return (cls + s) & 1; }
__host__ __device__ inline int orders_of(int cls, int s, int L) { return (L + 1 - first_order(cls, s)) / 2; }

Sets sets_of(int pass, int L, int s, int B, int pairs) {
  Sets q;
  for (int c = 0; c < 2; ++c) {
    q.n[c] = by_order(pass) ? 2 * B * orders_of(c, s, L) : B * L;
    q.tiles[c] = (q.n[c] + pairs - 1) / pairs;
  }
  return q;
}

__host__ __device__ inline int chunks_of(int L) { return (L + kChunkK - 1) / kChunkK; }

// ---------------------------------------------------------------------------------------------
// Matrices
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ double entry(int which, int L, const double2* cs, const double2* T, int r, int k) {
  if (r >= L || k >= L) return 0.0;
  const int n2 = 2 * (2 * L - 1);
  switch (which) {  // sin vanishes at the node theta = pi
    case kCosKX: return cs[(int)(((long long)k * (2 * r + 1)) % n2)].x;
    case kSinKX: return r == L - 1 ? 0.0 : cs[(int)(((long long)k * (2 * r + 1)) % n2)].y;
    case kCosXK: return cs[(int)(((long long)r * (2 * k + 1)) % n2)].x;
    case kSinXK: return k == L - 1 ? 0.0 : cs[(int)(((long long)r * (2 * k + 1)) % n2)].y;
    default: return weight_entry(which == kWeightE, L, cs, T, r, k);
  }
}

// A warp makes one row of one matrix (blockIdx.y): its exponent, then its digits.
__global__ void __launch_bounds__(128) digit_matrices_kernel(int L, const double2* __restrict__ cs, const double2* __restrict__ T,
                                                             uint8_t* __restrict__ out, int* __restrict__ exps) {
  const int lane = threadIdx.x & 31, r = blockIdx.x * 4 + (threadIdx.x >> 5), which = blockIdx.y;
  const int nc = chunks_of(L), rows = (L + 127) / 128 * 128;
  if (r >= rows) return;
  int e = 1;
  for (int k = lane; k < L; k += 32) e = max(e, exponent_of(entry(which, L, cs, T, r, k)));
  e = __reduce_max_sync(0xffffffffu, e);
  if (lane == 0) exps[which * rows + r] = e;
  uint8_t* t = out + ((size_t)which * (rows / 128) + (r >> 7)) * nc * kMatTile;
  for (int g = lane; g < 4 * nc; g += 32) {
    double x[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = entry(which, L, cs, T, r, 8 * g + k);
    put_digits<kDigits, 128 * 128>(t + (size_t)(g >> 2) * kMatTile, r & 127, g & 3, x, e);
  }
}

// ---------------------------------------------------------------------------------------------
// Data
// ---------------------------------------------------------------------------------------------
// A CTA takes kSources orders (theta passes) or rings (phi passes), each two complex columns -- four rows -- of
// all k: their largest exponents, then (read again above 512 k) their digits.  A thread takes eight k's of a
// source; the lanes run along whichever of k and source is contiguous.  Bound by latency at small batches
// and by HBM traffic (16 bytes written a value).
constexpr int kSources = 2, kPackThreads = 128;

struct PackArgs {
  int L, s, B;
  Sets q;
  const double2* in;
  long long in_n;
  uint8_t* x;
  int* exps;
};

template <int PASS>
__device__ __forceinline__ void load_pair(const PackArgs& a, int b, int i, int k, double2& u, double2& v) {
  const int L = a.L, N = 2 * L - 1;
  u = v = make_double2(0.0, 0.0);
  if (k >= L) return;
  auto at = [&](long long o) { return in_bounds(o, a.in_n, kbTorusIn) ? __ldg(&a.in[o]) : make_double2(0.0, 0.0); };
  if constexpr (PASS == kThetaInverse) {  // F [b][m + L - 1][m']: x_m +- x_{-m}
    const double2 x = at(((long long)b * N + L - 1 + i) * L + k);
    if (i == 0) {
      u = x;
    } else {
      const double2 y = at(((long long)b * N + L - 1 - i) * L + k);
      u = make_double2(x.x + y.x, x.y + y.y);
      v = make_double2(x.x - y.x, x.y - y.y);
    }
    if (k == 0) {  // the sum is doubled at the end
      u = make_double2(0.5 * u.x, 0.5 * u.y);
      v = make_double2(0.5 * v.x, 0.5 * v.y);
    }
  } else if constexpr (PASS == kPhiInverse) {  // E, O [2][b][m][t]
    const long long o = ((long long)b * L + k) * L + i;
    u = at(o);
    v = at(o + (long long)a.B * L * L);
  } else if constexpr (PASS == kPhiForward) {  // f [b][t][p], folded about the last node
    const long long o = ((long long)b * L + i) * N;
    const double2 x = at(o + k);
    if (k == L - 1) {
      u = x;
    } else {
      const double2 y = at(o + N - 1 - k);
      u = make_double2(x.x + y.x, x.y + y.y);
      v = make_double2(x.x - y.x, x.y - y.y);
    }
  } else {  // P, Q [2][b][t][m]: P -+ iQ
    const long long o = ((long long)b * L + k) * L + i;
    const double2 p = at(o), q = at(o + (long long)a.B * L * L);
    u = make_double2(p.x + q.y, p.y - q.x);
    v = make_double2(p.x - q.y, p.y + q.x);
  }
}

template <int PASS, int PAIRS>
__global__ void __launch_bounds__(kPackThreads) digit_pack_kernel(const __grid_constant__ PackArgs a) {
  __shared__ int top[kSources][4];
  constexpr bool along_k = PASS == kThetaInverse || PASS == kPhiForward;
  const int L = a.L, nc = chunks_of(L), groups = 4 * nc, items = kSources * groups;
  if (threadIdx.x < kSources * 4) top[threadIdx.x >> 2][threadIdx.x & 3] = 1;
  __syncthreads();
  double x[4][8];
  auto load = [&](int so, int g) {
    const long long src = (long long)blockIdx.x * kSources + so;
    if (src >= (long long)a.B * L) return false;
    const int b = (int)(src / L), i = (int)(src - (long long)b * L);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      double2 u, v;
      load_pair<PASS>(a, b, i, 8 * g + k, u, v);
      x[0][k] = u.x;
      x[1][k] = u.y;
      x[2][k] = v.x;
      x[3][k] = v.y;
    }
    return true;
  };
#pragma unroll 1
  for (int w = threadIdx.x; w < items; w += kPackThreads) {
    const int so = along_k ? w / groups : w % kSources, g = along_k ? w - so * groups : w / kSources;
    if (!load(so, g)) continue;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      int e = 1;
#pragma unroll
      for (int k = 0; k < 8; ++k) e = max(e, exponent_of(x[r][k]));
      if (e > *(volatile int*)&top[so][r]) atomicMax(&top[so][r], e);
    }
  }
  __syncthreads();
#pragma unroll 1
  for (int w = threadIdx.x; w < items; w += kPackThreads) {
    const int so = along_k ? w / groups : w % kSources, g = along_k ? w - so * groups : w / kSources;
    const long long src = (long long)blockIdx.x * kSources + so;
    if (src >= (long long)a.B * L) continue;
    if (items > kPackThreads) load(so, g);  // else its values are still here
    const int b = (int)(src / L), i = (int)(src - (long long)b * L);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      // set and column: both of an order's columns lie in its class, a ring's in one set each
      int set, col;
      if (by_order(PASS)) {
        set = (i + a.s) & 1;
        col = 2 * (b * orders_of(set, a.s, L) + (i >> 1)) + (r >> 1);
      } else {
        set = r >> 1;
        col = (int)src;
      }
      const int tile = (set ? a.q.tiles[0] : 0) + col / PAIRS, row = 2 * (col % PAIRS) + (r & 1), e = top[so][r];
      if (!in_bounds(tile, a.q.all(), kbTorusTile)) continue;
      if (g == 0) a.exps[tile * 2 * PAIRS + row] = e;
      put_digits<kDigits, 2 * PAIRS * 128>(a.x + ((size_t)tile * nc + (g >> 2)) * kDataTile<PAIRS>, row, g & 3, x[r], e);
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Products
// ---------------------------------------------------------------------------------------------
struct GemmArgs {
  int L, s, B;
  Sets q;
  int mblocks, ntiles;
  const uint8_t* A[2];
  const int* aexp[2];
  const uint8_t* x;
  const int* xexp;
  double2* out;
  long long out_n;
  int* status;
  long long wait_ns;
};

// Work item w: row block i, data tile j (of both sets in one count), set u.
struct Item {
  int i, j, u;
};
__device__ __forceinline__ Item item_of(const GemmArgs& a, int w) {
  Item t;
  t.i = w % a.mblocks;
  t.j = w / a.mblocks;
  t.u = t.j >= a.q.tiles[0];
  return t;
}

// Column of accumulator d: the even ones, then the odd ones.
template <int COLS>
__device__ __forceinline__ constexpr uint32_t acc_col(int d) { return COLS * (d >> 1) + (d & 1) * 4 * COLS; }

template <int PASS, int PAIRS>
__global__ void __launch_bounds__(kThreads, 1) digit_gemm_kernel(const __grid_constant__ GemmArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t full[kStages], empty[kStages], seg_full, seg_empty, done_bar;
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag;
  constexpr int STAGE = kStageBytes<PAIRS>, DATA = kDataTile<PAIRS>, COLS = 2 * PAIRS, PER = COLS / 4;  // columns of a thread
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp == 1) tmem_alloc(&tmem_base, kDigits * COLS);
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(&seg_full, 1);
    mbar_init(&seg_empty, kEpiWarps);
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
      // ---- producer ----
      const bool one = elect_one();
      int s = 0, ph = 1;
      uint32_t used = 0, uph = 0;  // stages that were filled, and the parity of their last fill
      for (int w = blockIdx.x; w < a.ntiles && going(abort); w += gridDim.x) {
        const Item t = item_of(a, w);
        // (a tile outside its array is recorded and the first one copied instead: the pipeline still completes)
        const bool here = in_bounds(t.i, a.mblocks, kbDigitTile) && in_bounds(t.j, a.q.all(), kbDigitTile);
        const uint8_t* m = a.A[t.u] + (size_t)(here ? t.i : 0) * nc * kMatTile;
        const uint8_t* x = a.x + (size_t)(here ? t.j : 0) * nc * DATA;
        for (int c = 0; c < nc; ++c) {
          if (!__all_sync(0xffffffffu, mbar_wait(&empty[s], ph, abort, a.wait_ns))) {
            *abort = 1;
            break;
          }
          if (one) {
            uint8_t* st = smem + s * STAGE;
            mbar_expect_tx(&full[s], (uint32_t)STAGE);
            bulk_g2s(st, m + (size_t)c * kMatTile, kMatTile, &full[s]);
            bulk_g2s(st + kMatTile, x + (size_t)c * DATA, DATA, &full[s]);
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
        if ((used >> k) & 1u) mbar_wait(&full[k], (uph >> k) & 1u, nullptr, kDrainNs);
    } else if (warp == 1) {
      // ---- MMA issuer: per 16 k's the 36 digit products, digits i + j into accumulator i + j.  A part of the data
      // tile holds two digits, so the even (or the odd) ones are the rows of one operand, and with the accumulators of one parity
      // side by side one product takes digit i of the matrix times all of them ----
      const bool one = elect_one();
      const uint32_t lo0 = (smem_u32(smem) >> 4) + kDescLow;
      int s = 0, ph = 0, sph = 1;
      for (int w = blockIdx.x; w < a.ntiles && going(abort); w += gridDim.x)
        for (int c = 0; c < nc; ++c) {
          const bool first = c % kSegChunks == 0, last = c + 1 == nc || (c + 1) % kSegChunks == 0;
          const bool here = (!first || mbar_wait(&seg_empty, sph, abort, a.wait_ns)) && mbar_wait(&full[s], ph, abort, a.wait_ns);
          if (!__all_sync(0xffffffffu, here)) {
            *abort = 1;
            break;
          }
          if (first) sph ^= 1;
          fence_after();
          if (one) {
            const uint32_t la = lo0 + (uint32_t)(s * (STAGE >> 4)), lb = la + (kMatTile >> 4);
#pragma unroll
            for (int kk = 0; kk < 2; ++kk)
#pragma unroll
              for (int i = 0; i < kDigits; ++i) {
                const int jm = kDigits - 1 - i, even = jm / 2 + 1, odd = (jm + 1) / 2;
                const uint32_t da = la + (i >> 1) * (128 * 128 >> 4) + (i & 1) * 4 + 2 * kk, init = first && kk == 0 && i == 0 ? 0u : 1u;
                mma_f16_lo<false>(tbase + acc_col<COLS>(i), da, lb + 2 * kk, idesc_f16(128, COLS * even), init);
                if (odd) mma_f16_lo<false>(tbase + acc_col<COLS>(i + 1), da, lb + 4 + 2 * kk, idesc_f16(128, COLS * odd), init);
              }
            mma_commit(&empty[s]);
            if (last) mma_commit(&seg_full);
          }
          __syncwarp();
          if (++s == kStages) {
            s = 0;
            ph ^= 1;
          }
        }
      // every issued product has completed before the CTA leaves
      if (one) mma_commit(&done_bar);
      __syncwarp();
      mbar_wait(&done_bar, 0, nullptr, kDrainNs);
    }
  } else {
    // ---- epilogue: a thread has one row, PER columns (PER / 2 complex ones) ----
    regs_inc<kRegsEpilogue>();
    const int q = warp & 3, cg = (warp - 4) >> 2;
    const uint32_t tq = tbase + ((uint32_t)(q * 32) << 16) + PER * cg;
    int ph = 0;
    for (int w = blockIdx.x; w < a.ntiles && going(abort); w += gridDim.x) {
      const Item t = item_of(a, w);
      long long hi[PER], lo[PER];
#pragma unroll
      for (int k = 0; k < PER; ++k) hi[k] = lo[k] = 0;
      bool ok = true;
      for (int c0 = 0; c0 < nc; c0 += kSegChunks) {
        if (!__all_sync(0xffffffffu, mbar_wait(&seg_full, ph, abort, a.wait_ns))) {
          *abort = 1;
          ok = false;
          break;
        }
        ph ^= 1;
        fence_after();
#pragma unroll
        for (int h = 0; h < PER / 8; ++h)
#pragma unroll
          for (int d = 0; d < kDigits; d += 4) {
            int v[4][8];
#pragma unroll
            for (int k = 0; k < 4; ++k) tmem_ld8_nowait(tq + acc_col<COLS>(d + k) + 8 * h, (uint32_t*)v[k]);
            tmem_wait_ld();
            // whole numbers of at most (d + 1) 2^21: the pairs' sums stay below 2^31
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              const int x = __float2int_rn(__int_as_float(v[0][k])) * 128 + __float2int_rn(__int_as_float(v[1][k]));
              const int y = __float2int_rn(__int_as_float(v[2][k])) * 128 + __float2int_rn(__int_as_float(v[3][k]));
              (d ? lo : hi)[8 * h + k] += (long long)x * 16384 + y;
            }
          }
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&seg_empty);
      }
      if (!ok) break;
      const int row = t.i * 128 + q * 32 + lane;
      const int col0 = (t.j - (t.u ? a.q.tiles[0] : 0)) * PAIRS + PER / 2 * cg;
      if (row >= L || !in_bounds(row, 128 * a.mblocks, kbDigitExp) || !in_bounds(t.j, a.q.all(), kbDigitExp)) continue;
      const int ea = a.aexp[t.u][row] - 2105;
      const int* xe = a.xexp + (size_t)t.j * COLS + PER * cg;
#pragma unroll
      for (int k = 0; k < PER / 2; ++k) {
        const int col = col0 + k;
        if (col >= a.q.n[t.u]) break;
        const int2 e = __ldg((const int2*)xe + k);
        const int twice = PASS == kThetaInverse || (PASS == kThetaAdjoint && row > 0) ? 1 : 0;
        double2 z = make_double2(assemble(hi[2 * k], lo[2 * k], ea + e.x + twice), assemble(hi[2 * k + 1], lo[2 * k + 1], ea + e.y + twice));
        if constexpr (PASS == kPhiInverse || PASS == kPhiForward) {
          const long long o = ((long long)t.u * a.B * L + col) * L + row;
          if (in_bounds(o, a.out_n, kbTorusOut)) a.out[o] = z;
        } else {
          const int second = col & 1, no = orders_of(t.u, a.s, L), b = (col >> 1) / no;
          const int m = 2 * ((col >> 1) - b * no) + first_order(t.u, a.s);
          if constexpr (PASS == kThetaInverse) {
            const long long o = (((long long)second * a.B + b) * L + m) * L + row;
            if (t.u) z = make_double2(-z.y, z.x);  // times i
            if (in_bounds(o, a.out_n, kbTorusOut)) a.out[o] = z;
          } else {
            const long long o = ((long long)b * (2 * L - 1) + L - 1 + (second ? -m : m)) * L + row;
            if (t.u) z = make_double2(z.y, -z.x);  // times -i
            if ((!second || m > 0) && in_bounds(o, a.out_n, kbTorusOut)) a.out[o] = z;
          }
        }
      }
    }
  }
  fence_before();
  __syncthreads();
  fence_after();
  if (*abort && threadIdx.x == 0) atomicOr(a.status, 2);
  if (warp == 1) tmem_dealloc(tbase, kDigits * COLS);
}

// phi of the inverse: C, S [2][b][t][p] -> f[b][t][p] = C + iS, f[b][t][N - 1 - p] = C - iS.
__global__ void __launch_bounds__(256) digit_join_kernel(int L, long long rings, const double2* __restrict__ cs, long long cs_n,
                                                         double2* __restrict__ f, long long f_n) {
  const long long e = (long long)blockIdx.x * 256 + threadIdx.x;
  if (e >= rings * L) return;
  const long long r = e / L, o = r * (2 * L - 1);
  const int p = (int)(e - r * L);
  if (!in_bounds(e + rings * L, cs_n, kbTorusIn) || !in_bounds(o + p, f_n, kbTorusOut)) return;
  const double2 c = __ldg(&cs[e]), z = __ldg(&cs[e + rings * L]);
  f[o + p] = make_double2(c.x - z.y, c.y + z.x);
  if (p < L - 1) f[o + 2 * L - 2 - p] = make_double2(c.x + z.y, c.y - z.x);
}

}  // namespace

struct DigitPlan {
  int L = 0, sms = 0;
  uint8_t* mats = nullptr;
  int* exps = nullptr;
  size_t bytes = 0;
};

size_t digits_workspace_bytes(int L, int s, int B) {
  size_t n = 0;
  for (int pass : {(int)kThetaInverse, (int)kPhiInverse}) {
    const size_t t = sets_of(pass, L, s, B, 32).all();  // tiles of 16 pad less
    n = std::max(n, t * chunks_of(L) * kDataTile<32> + t * 64 * sizeof(int));
  }
  return n;
}

template <int PASS>
static cudaError_t pass_attr() {
  cudaError_t e = prefer_shared(digit_gemm_kernel<PASS, 32>);
  if (e == cudaSuccess) e = prefer_shared(digit_gemm_kernel<PASS, 16>);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(digit_gemm_kernel<PASS, 32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem<32>);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(digit_gemm_kernel<PASS, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem<16>);
  return e;
}

cudaError_t digits_setup(DigitPlan** out, int L, int device) {
  *out = nullptr;
  DigitPlan* p = new DigitPlan();
  p->L = L;
  const int rows = (L + 127) / 128 * 128;
  const size_t ncs = 2 * (size_t)(2 * L - 1), n = (size_t)L * L;
  const size_t mats = (size_t)kMatrices * (rows / 128) * chunks_of(L) * kMatTile, exps = (size_t)kMatrices * rows * sizeof(int);
  double2* tmp = nullptr;
  cudaError_t e = cudaDeviceGetAttribute(&p->sms, cudaDevAttrMultiProcessorCount, device);
  if (e == cudaSuccess) e = pass_attr<kThetaInverse>();
  if (e == cudaSuccess) e = pass_attr<kPhiInverse>();
  if (e == cudaSuccess) e = pass_attr<kPhiForward>();
  if (e == cudaSuccess) e = pass_attr<kThetaForward>();
  if (e == cudaSuccess) e = pass_attr<kThetaAdjoint>();
  if (e == cudaSuccess) e = dev_malloc(&p->mats, mats);
  if (e == cudaSuccess) e = dev_malloc(&p->exps, exps);
  if (e == cudaSuccess) {
    p->bytes = mats + exps;
    e = dev_malloc(&tmp, (ncs + n) * sizeof(double2));
  }
  if (e == cudaSuccess) {
    node_table_kernel<<<(unsigned)((ncs + 255) / 256), 256>>>(2 * L - 1, tmp);
    weight_prefix_kernel<<<(unsigned)((L + 31) / 32), 32>>>(L, tmp, tmp + ncs);
    digit_matrices_kernel<<<dim3(rows / 4, kMatrices), 128>>>(L, tmp, tmp + ncs, p->mats, p->exps);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
  }
  if (tmp) cudaFree(tmp);
  if (e != cudaSuccess) {
    digits_destroy(p);
    return e;
  }
  *out = p;
  return cudaSuccess;
}

void digits_destroy(DigitPlan* p) {
  if (!p) return;
  if (p->mats) cudaFree(p->mats);
  if (p->exps) cudaFree(p->exps);
  delete p;
}

size_t digits_bytes(const DigitPlan* p) { return p ? p->bytes : 0; }

template <int PASS, int PAIRS>
static cudaError_t run_tiles(const DigitPlan* p, int mat, int s, int B, const void* in, size_t in_bytes, void* work,
                             size_t work_bytes, void* out, size_t out_bytes, int* status, long long wait_ns, cudaStream_t st) {
  const int L = p->L, rows = (L + 127) / 128 * 128;
  const Sets q = sets_of(PASS, L, s, B, PAIRS);
  const size_t tile_bytes = (size_t)q.all() * chunks_of(L) * kDataTile<PAIRS>;
  if (tile_bytes + (size_t)q.all() * 2 * PAIRS * sizeof(int) > work_bytes) return cudaErrorInvalidValue;
  PackArgs k{};
  k.L = L;
  k.s = s;
  k.B = B;
  k.q = q;
  k.in = (const double2*)in;
  k.in_n = (long long)(in_bytes / sizeof(double2));
  k.x = (uint8_t*)work;
  k.exps = (int*)((uint8_t*)work + tile_bytes);
  digit_pack_kernel<PASS, PAIRS><<<(unsigned)(((long long)B * L + kSources - 1) / kSources), kPackThreads, 0, st>>>(k);
  GemmArgs a{};
  a.L = L;
  a.s = s;
  a.B = B;
  a.q = q;
  a.mblocks = rows / 128;
  a.ntiles = a.mblocks * q.all();
  for (int u = 0; u < 2; ++u) {
    a.A[u] = p->mats + (size_t)(mat + u) * a.mblocks * chunks_of(L) * kMatTile;
    a.aexp[u] = p->exps + (mat + u) * rows;
  }
  a.x = k.x;
  a.xexp = k.exps;
  a.out = (double2*)out;
  a.out_n = (long long)(out_bytes / sizeof(double2));
  a.status = status;
  a.wait_ns = wait_ns;
  digit_gemm_kernel<PASS, PAIRS><<<(unsigned)std::min(a.ntiles, p->sms), kThreads, kSmem<PAIRS>, st>>>(a);
  return cudaGetLastError();
}

// Tiles of 16 complex columns where those of 32 would leave half of the SMs without one: L = 129, B = 4 (66 and
// 130 tiles) 21.8 us a product with 32, 17.4 with 16 (13.5 since the digits are taken together).
template <int PASS>
static cudaError_t run(const DigitPlan* p, int mat, int s, int B, const void* in, size_t in_bytes, void* work,
                             size_t work_bytes, void* out, size_t out_bytes, int* status, long long wait_ns, cudaStream_t st) {
  const int tiles = (p->L + 127) / 128 * sets_of(PASS, p->L, s, B, 32).all();
  return 2 * tiles <= p->sms ? run_tiles<PASS, 16>(p, mat, s, B, in, in_bytes, work, work_bytes, out, out_bytes, status, wait_ns, st)
                             : run_tiles<PASS, 32>(p, mat, s, B, in, in_bytes, work, work_bytes, out, out_bytes, status, wait_ns, st);
}

cudaError_t digits_pass(const DigitPlan* p, int which, int s, int B, const void* in, size_t in_bytes, void* work,
                        size_t work_bytes, void* mid, size_t mid_bytes, void* out, size_t out_bytes, int* status, long long wait_ns, cudaStream_t st) {
  switch (which) {
    case kThetaInverse: return run<kThetaInverse>(p, kCosKX, s, B, in, in_bytes, work, work_bytes, out, out_bytes, status, wait_ns, st);
    case kPhiForward: return run<kPhiForward>(p, kCosXK, s, B, in, in_bytes, work, work_bytes, out, out_bytes, status, wait_ns, st);
    case kThetaForward: return run<kThetaForward>(p, kWeightE, s, B, in, in_bytes, work, work_bytes, out, out_bytes, status, wait_ns, st);
    case kThetaAdjoint: return run<kThetaAdjoint>(p, kCosXK, s, B, in, in_bytes, work, work_bytes, out, out_bytes, status, wait_ns, st);
    default: break;
  }
  cudaError_t e = run<kPhiInverse>(p, kCosKX, s, B, in, in_bytes, work, work_bytes, mid, mid_bytes, status, wait_ns, st);
  if (e != cudaSuccess) return e;
  const long long rings = (long long)B * p->L;
  digit_join_kernel<<<(unsigned)((rings * p->L + 255) / 256), 256, 0, st>>>(p->L, rings, (const double2*)mid,
                                                                           (long long)(mid_bytes / sizeof(double2)), (double2*)out,
                                                                           (long long)(out_bytes / sizeof(double2)));
  return cudaGetLastError();
}

SSHT_BOUNDS_TU(torus_digits)

}  // namespace ssht
