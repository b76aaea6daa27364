// Torus passes of FP64 plans with little work: the folded cosine and sine products of the torus stage
// (torus_gemm.cu gives the identities) in FP64 on CUDA cores, four launches an inverse + forward.
//
// Matrices are stored [k][row], so that a warp's lanes (32 rows) read them coalesced, and a data column is
// read by the whole warp at one address.  A CTA computes 32 rows of one unit -- one order |m| (both signs), or
// one ring -- as two complex columns, 4 FP64 multiply-adds a k; its eight warps take an eighth of the k's each
// and add up at the end, which keeps every quarter of every SM busy down to the smallest band-limits.
//
// What bounds it: launches and latency at the smallest sizes, then the FP64 pipe, 8 B L^3 flops a pass
// (1.07 TFLOP/s at L = 128, B = 16, 0.85 of its rate).  L = 64, B = 1: 43 us, by FFTs 141.
#include "bounds.cuh"
#include "ssht_internal.h"
#include "torus_matrices.cuh"

#include <algorithm>

namespace ssht {
namespace {

constexpr int kWarps = 8;

using namespace folded;

struct Pair {
  double2 a, b;
};

// Sum of the eight warps' pairs for lane's row, in warp 0 (all threads call it).
__device__ __forceinline__ Pair reduce_warps(Pair v, int warp, int lane) {
  __shared__ double2 part[kWarps][2][32];
  part[warp][0][lane] = v.a;
  part[warp][1][lane] = v.b;
  __syncthreads();
  Pair r;
  r.a = r.b = make_double2(0.0, 0.0);
  if (warp == 0)
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const double2 a = part[w][0][lane], b = part[w][1][lane];
      r.a.x += a.x;
      r.a.y += a.y;
      r.b.x += b.x;
      r.b.y += b.y;
    }
  return r;
}

// Element i of a run that starts `at` elements into a buffer of n, zero outside (checked builds).
__device__ __forceinline__ double2 load(const double2* run, size_t i, size_t at, long long n) {
  return in_bounds((long long)(at + i), n, kbTorusIn) ? __ldg(&run[i]) : make_double2(0.0, 0.0);
}
__device__ __forceinline__ void store(double2* run, size_t i, size_t at, long long n, double2 v) {
  if (in_bounds((long long)(at + i), n, kbTorusOut)) run[i] = v;
}

__device__ __forceinline__ void axpy(double2& acc, double a, double2 x) {
  acc.x = fma(a, x.x, acc.x);
  acc.y = fma(a, x.y, acc.y);
}

// theta inverse: F [b][m + Lp][m'] -> work E, O [2][b][m][t] = x_m +- x_{-m} (m = 0: x_0, 0).
__global__ void __launch_bounds__(32 * kWarps) direct_theta_inverse_kernel(int L, int s, int B, const double* __restrict__ M,
                                                                           const double2* __restrict__ F, long long in_n,
                                                                           double2* __restrict__ work, long long out_n) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, N = 2 * L - 1;
  const int t = 32 * blockIdx.y + lane, b = blockIdx.x / L, m = blockIdx.x - b * L;
  const bool odd = (m + s) & 1;
  const double* A = M + (size_t)(odd ? kSinKX : kCosKX) * L * L;
  const size_t fp = ((size_t)b * N + L - 1 + m) * L, fm = ((size_t)b * N + L - 1 - m) * L;
  const double2* Fp = F + fp;
  const double2* Fm = F + fm;
  Pair v;
  v.a = v.b = make_double2(0.0, 0.0);
#pragma unroll 4
  for (int k = warp; k < L; k += kWarps) {
    double a = t < L ? __ldg(&A[(size_t)k * L + t]) : 0.0;
    if (k == 0) a *= 0.5;  // the sum is doubled below
    axpy(v.a, a, load(Fp, k, fp, in_n));
    axpy(v.b, a, load(Fm, k, fm, in_n));
  }
  v = reduce_warps(v, warp, lane);
  if (warp || t >= L) return;
  double2 e = v.a, o = make_double2(0.0, 0.0);
  if (m > 0) {
    e = make_double2(v.a.x + v.b.x, v.a.y + v.b.y);
    o = make_double2(v.a.x - v.b.x, v.a.y - v.b.y);
  }
  if (odd) {  // times i
    e = make_double2(-e.y, e.x);
    o = make_double2(-o.y, o.x);
  }
  const size_t at = ((size_t)b * L + m) * L + t;
  store(work, at, 0, out_n, make_double2(2.0 * e.x, 2.0 * e.y));
  store(work, (size_t)B * L * L + at, 0, out_n, make_double2(2.0 * o.x, 2.0 * o.y));
}

// phi inverse: E, O [2][b][m][t] -> f[b][t][p] = E + iO, f[b][t][N-1-p] = E - iO.
__global__ void __launch_bounds__(32 * kWarps) direct_phi_inverse_kernel(int L, int B, const double* __restrict__ M,
                                                                         const double2* __restrict__ work, long long in_n,
                                                                         double2* __restrict__ f, long long out_n) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, N = 2 * L - 1;
  const int p = 32 * blockIdx.y + lane, b = blockIdx.x / L, t = blockIdx.x - b * L;
  const double* C = M + (size_t)kCosKX * L * L;
  const double* S = M + (size_t)kSinKX * L * L;
  const size_t e0 = (size_t)b * L * L + t, o0 = e0 + (size_t)B * L * L;
  const double2* E = work + e0;
  const double2* O = work + o0;
  Pair v;
  v.a = v.b = make_double2(0.0, 0.0);
#pragma unroll 4
  for (int k = warp; k < L; k += kWarps) {
    const double c = p < L ? __ldg(&C[(size_t)k * L + p]) : 0.0, sn = p < L ? __ldg(&S[(size_t)k * L + p]) : 0.0;
    axpy(v.a, c, load(E, (size_t)k * L, e0, in_n));
    axpy(v.b, sn, load(O, (size_t)k * L, o0, in_n));
  }
  v = reduce_warps(v, warp, lane);
  if (warp || p >= L) return;
  const size_t r0 = ((size_t)b * L + t) * N;
  double2* row = f + r0;
  store(row, p, r0, out_n, make_double2(v.a.x - v.b.y, v.a.y + v.b.x));
  if (p < L - 1) store(row, N - 1 - p, r0, out_n, make_double2(v.a.x + v.b.y, v.a.y - v.b.x));
}

// phi of forward and adjoint: f [b][t][p] -> P, Q [2][b][t][m].  A warp folds 32 of its k's at a time.
__global__ void __launch_bounds__(32 * kWarps) direct_phi_forward_kernel(int L, int B, const double* __restrict__ M,
                                                                         const double2* __restrict__ f, long long in_n,
                                                                         double2* __restrict__ work, long long out_n) {
  __shared__ double2 fold[kWarps][2][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, N = 2 * L - 1;
  const int m = 32 * blockIdx.y + lane, b = blockIdx.x / L, t = blockIdx.x - b * L;
  const double* C = M + (size_t)kCosXK * L * L;
  const double* S = M + (size_t)kSinXK * L * L;
  const size_t r0 = ((size_t)b * L + t) * N;
  const double2* row = f + r0;
  const int per = (L + kWarps - 1) / kWarps, k_end = min(L, (warp + 1) * per);
  Pair v;
  v.a = v.b = make_double2(0.0, 0.0);
  for (int k0 = warp * per; k0 < k_end; k0 += 32) {
    const int p = k0 + lane;
    double2 e = make_double2(0.0, 0.0), o = e;
    if (p < k_end) {
      e = load(row, p, r0, in_n);
      if (p < L - 1) {
        const double2 y = load(row, N - 1 - p, r0, in_n);
        o = make_double2(e.x - y.x, e.y - y.y);
        e = make_double2(e.x + y.x, e.y + y.y);
      }
    }
    __syncwarp();
    fold[warp][0][lane] = e;
    fold[warp][1][lane] = o;
    __syncwarp();
    const int n = min(32, k_end - k0);
#pragma unroll 4
    for (int i = 0; i < n; ++i) {
      const double c = m < L ? __ldg(&C[(size_t)(k0 + i) * L + m]) : 0.0, sn = m < L ? __ldg(&S[(size_t)(k0 + i) * L + m]) : 0.0;
      axpy(v.a, c, fold[warp][0][i]);
      axpy(v.b, sn, fold[warp][1][i]);
    }
  }
  v = reduce_warps(v, warp, lane);
  if (warp || m >= L) return;
  const size_t at = ((size_t)b * L + t) * L + m;
  store(work, at, 0, out_n, v.a);
  store(work, (size_t)B * L * L + at, 0, out_n, v.b);
}

// theta of forward (weight matrices) and adjoint (cosines and sines, the fold of m' < 0): P, Q -> H [b][m + Lp][m'].
__global__ void __launch_bounds__(32 * kWarps) direct_theta_forward_kernel(int L, int s, int B, int adjoint,
                                                                           const double* __restrict__ M,
                                                                           const double2* __restrict__ work, long long in_n,
                                                                           double2* __restrict__ H, long long out_n) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, N = 2 * L - 1;
  const int mp = 32 * blockIdx.y + lane, b = blockIdx.x / L, m = blockIdx.x - b * L;
  const bool odd = (m + s) & 1;
  const double* A = M + (size_t)(adjoint ? (odd ? kSinXK : kCosXK) : (odd ? kWeightO : kWeightE)) * L * L;
  const size_t p0 = (size_t)b * L * L + m, q0 = p0 + (size_t)B * L * L;
  const double2* P = work + p0;
  const double2* Q = work + q0;
  Pair v;
  v.a = v.b = make_double2(0.0, 0.0);
#pragma unroll 4
  for (int k = warp; k < L; k += kWarps) {
    const double a = mp < L ? __ldg(&A[(size_t)k * L + mp]) : 0.0;
    axpy(v.a, a, load(P, (size_t)k * L, p0, in_n));
    axpy(v.b, a, load(Q, (size_t)k * L, q0, in_n));
  }
  v = reduce_warps(v, warp, lane);
  if (warp || mp >= L) return;
  const double w = adjoint && mp > 0 ? 2.0 : 1.0;
  double2 hp = make_double2(w * (v.a.x + v.b.y), w * (v.a.y - v.b.x)), hm = make_double2(w * (v.a.x - v.b.y), w * (v.a.y + v.b.x));
  if (odd) {  // times -i
    hp = make_double2(hp.y, -hp.x);
    hm = make_double2(hm.y, -hm.x);
  }
  store(H, ((size_t)b * N + L - 1 + m) * L + mp, 0, out_n, hp);
  if (m > 0) store(H, ((size_t)b * N + L - 1 - m) * L + mp, 0, out_n, hm);
}

}  // namespace

struct DirectPlan {
  int L = 0;
  double* mats = nullptr;
  size_t bytes = 0;
};

// Where these products beat those of digits: for little work, where the digits' nine launches set the time, and
// at band-limits that fill little of their tiles (many fields of those take torus_small.cu).  GB300, torus stage of an inverse
// and a forward in us, digits against these: L = 64, B = 1 95 and 43; L = 96, B = 1 101 and 56; L = 128, B = 1 107 and 102;
// L = 32, B = 128 193 and 185; beyond the line L = 96, B = 2 104 and 85, L = 64, B = 8 98 and 103 (the two meet there); L = 144,
// B = 1 115 and 132; L = 128, B = 4 114 and 283.
bool direct_wanted(int L, int B) { return L <= 32 || (long long)B * L * L * L <= (1ll << 21); }

cudaError_t direct_setup(DirectPlan** out, int L) {
  *out = nullptr;
  DirectPlan* p = new DirectPlan();
  p->L = L;
  const cudaError_t e = make_matrices(L, &p->mats, &p->bytes);
  if (e != cudaSuccess) {
    direct_destroy(p);
    return e;
  }
  *out = p;
  return cudaSuccess;
}

void direct_destroy(DirectPlan* p) {
  if (!p) return;
  if (p->mats) cudaFree(p->mats);
  delete p;
}

size_t direct_bytes(const DirectPlan* p) { return p ? p->bytes : 0; }

cudaError_t direct_inverse(const DirectPlan* p, int s, int B, const void* in, size_t in_bytes, void* out, size_t out_bytes,
                           cudaStream_t st, int step) {
  const dim3 grid((unsigned)B * p->L, (p->L + 31) / 32);
  const long long in_n = (long long)(in_bytes / sizeof(double2)), out_n = (long long)(out_bytes / sizeof(double2));
  if (step == 0)
    direct_theta_inverse_kernel<<<grid, 32 * kWarps, 0, st>>>(p->L, s, B, p->mats, (const double2*)in, in_n, (double2*)out, out_n);
  else
    direct_phi_inverse_kernel<<<grid, 32 * kWarps, 0, st>>>(p->L, B, p->mats, (const double2*)in, in_n, (double2*)out, out_n);
  return cudaGetLastError();
}

cudaError_t direct_analysis(const DirectPlan* p, int adjoint, int s, int B, const void* in, size_t in_bytes, void* out,
                            size_t out_bytes, cudaStream_t st, int step) {
  const dim3 grid((unsigned)B * p->L, (p->L + 31) / 32);
  const long long in_n = (long long)(in_bytes / sizeof(double2)), out_n = (long long)(out_bytes / sizeof(double2));
  if (step == 0)
    direct_phi_forward_kernel<<<grid, 32 * kWarps, 0, st>>>(p->L, B, p->mats, (const double2*)in, in_n, (double2*)out, out_n);
  else
    direct_theta_forward_kernel<<<grid, 32 * kWarps, 0, st>>>(p->L, s, B, adjoint, p->mats, (const double2*)in, in_n, (double2*)out,
                                                              out_n);
  return cudaGetLastError();
}

SSHT_BOUNDS_TU(torus_direct)

}  // namespace ssht
