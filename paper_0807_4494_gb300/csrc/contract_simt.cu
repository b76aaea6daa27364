// The O(L^3) contractions on CUDA cores, FP64 (and FP32 data with the same code).
//
// Inverse (eqn fourier_coeff, Sec. 3.1), for m' >= 0:
//   F_{m m'} = (-1)^s i^{-(m+s)} sum_{l >= max(|m|, m', |s|)} U_l[m'] Delta^l_{m' m} sf_lm,
//   U_l[m'] = sqrt((2l+1)/4pi) Delta^l_{m',-s}.
// Both signs of m share the products U Delta (Delta^l_{m',-m} = (-1)^{l+m'} Delta^l_{m' m}, eqn
// wignerd_sym6), and so do the fields of a thread.
//
// Projection (forward transform and adjoint), for l >= |s|:
//   sf_lm = (-1)^s i^{m+s} sum_{m'=0}^{l} U_l[m'] Delta^l_{m' m} H_{m m'}
// where H already folds the m' < 0 half (H_{m m'} = G_{m m'} + (-1)^{m+s} G_{m,-m'}).
//
// Both read the quadrant table's row m of degree l, contiguous in m', through
// Delta^l_{m' m} = (-1)^{m'-m} Delta^l_{m m'}, 32 values a warp.
//
// What bounds them: the FP64 pipe (2 lanes an SM and clock, so that a warp's instruction holds its
// quarter of the SM for 64 clocks): a product U Delta and 4 multiply-adds a field an entry, 0.38 ms a
// direction at L = 512 with one field.  Work is therefore cut so fine that every quarter of every SM has
// some: the inverse takes a CTA for 32 m' of one order, its eight warps taking every eighth degree
// each and adding up at the end; the projection a warp for a few degrees of one order, whose
// sums over the lanes are closed together (halving the values and the lanes at once: one addition a value
// instead of five).  GB300, against one thread an (order, m') over all degrees and one warp a (degree, order),
// inverse and projection: FP64 L = 512, B = 1 828 and 1344 -> 529 and 485 us, L = 129, B = 4 169 and 126 -> 44 and
// 51, FP32 L = 256, B = 8 225 and 541 -> 100 and 126.
#include "ssht_internal.h"
#include "bounds.cuh"
#include "f32_round.h"

namespace ssht {
namespace {

template <typename T> struct Cplx;
template <> struct Cplx<double> { using type = double2; };
template <> struct Cplx<float> { using type = float2; };

__host__ __device__ __forceinline__ long long tri_ll(long long m) { return m * (m + 1) / 2; }
__host__ __device__ __forceinline__ size_t doff(long long l) { return (size_t)(l * (l + 1) * (2 * l + 1) / 6); }

// (-1)^{s + e} i^k (x, y): parts exchanged and signs flipped, no arithmetic
template <typename C, typename T>
__device__ __forceinline__ C times_ik(int s, int e, int k, T x, T y) {
  const int r = ((k + 2 * (s + e)) % 4 + 4) % 4;
  C v;
  v.x = r == 0 ? x : r == 1 ? -y : r == 2 ? -x : y;
  v.y = r == 0 ? y : r == 1 ? x : r == 2 ? -y : -x;
  return v;
}

// The product U Delta, rounded once to the element type (FP32 by integer operations: f32_round.h).
template <typename T> __device__ __forceinline__ T ud(double u, double d);
template <> __device__ __forceinline__ double ud<double>(double u, double d) { return u * d; }
template <> __device__ __forceinline__ float ud<float>(double u, double d) { return f64_to_f32_rn(u * d); }

constexpr int kWarps = 8;

// One CTA: order |m| = blockIdx.y, m' = 32 blockIdx.x + lane, FB fields (blockIdx.z); warp w takes the
// degrees lmin + w, lmin + w + 8, ...
template <typename T, int FB>
__global__ void __launch_bounds__(32 * kWarps) inverse_kernel(int L, int s, int B, const double* __restrict__ table,
                                                              const double* __restrict__ U,
                                                              const typename Cplx<T>::type* __restrict__ flm,
                                                              typename Cplx<T>::type* __restrict__ E,
                                                              long long in_n, long long out_n) {
  using C = typename Cplx<T>::type;
  __shared__ C part[kWarps][2 * FB][32];
  const int Lp = L - 1, N = 2 * L - 1;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int m = blockIdx.y, mp0 = 32 * blockIdx.x, mp = mp0 + lane, b0 = blockIdx.z * FB;
  const int as = s < 0 ? -s : s;
  const int lmin = max(max(m, mp0), as);  // the lanes of larger m' join at l = m'
  C acc[2 * FB];
#pragma unroll
  for (int j = 0; j < 2 * FB; ++j) acc[j].x = acc[j].y = T(0);
#pragma unroll 2
  for (int l = lmin + warp; l <= Lp; l += kWarps) {
    T t = T(0);
    if (mp <= l) t = ud<T>(__ldg(&U[tri_ll(l) + mp]), __ldg(&table[doff(l) + (size_t)m * (l + 1) + mp]));
    const T tn = (l & 1) ? -t : t;  // (-1)^l for -m
    const long long cp = (long long)b0 * L * L + (long long)l * l + l + m;
#pragma unroll
    for (int j = 0; j < FB; ++j) {
      C a, an;
      a.x = a.y = an.x = an.y = T(0);
      if (b0 + j < B) {
        const long long ip = cp + (long long)j * L * L, in = ip - 2 * m;
        if (in_bounds(ip, in_n, kbSimtIn)) a = flm[ip];
        if (in_bounds(in, in_n, kbSimtIn)) an = flm[in];
      }
      acc[2 * j].x = fma(t, a.x, acc[2 * j].x);
      acc[2 * j].y = fma(t, a.y, acc[2 * j].y);
      acc[2 * j + 1].x = fma(tn, an.x, acc[2 * j + 1].x);
      acc[2 * j + 1].y = fma(tn, an.y, acc[2 * j + 1].y);
    }
  }
#pragma unroll
  for (int j = 0; j < 2 * FB; ++j) part[warp][j][lane] = acc[j];
  __syncthreads();
  // the warps' sums and outputs: one (field, sign) a warp
  for (int j = warp; j < 2 * FB; j += kWarps) {
    const int b = b0 + (j >> 1), sgn = j & 1;
    if (b >= B || mp > Lp || (sgn && m == 0)) continue;
    T ar = T(0), ai = T(0);
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      ar += part[w][j][lane].x;
      ai += part[w][j][lane].y;
    }
    const int mm = sgn ? -m : m;
    // +m: (-1)^{m'-m}; -m: (-1)^m (the row m of the table stands for Delta_{m' m})
    const C F = times_ik<C>(s, sgn ? m : mp - m, -(mm + s), ar, ai);
    const long long o = ((long long)b * N + (mm + Lp)) * L + mp;
    if (in_bounds(o, out_n, kbSimtOut)) E[o] = F;
  }
}

// Sums of NV values over the warp's lanes, all at once: every step sends half of the values to the
// partner lane and adds the other half, so that lane r ends with the sum of value index r >> (5 - log2 NV).
template <typename T, int NV>
__device__ __forceinline__ T warp_sums(T (&v)[NV], int lane) {
  int w = 16;
#pragma unroll
  for (int n = NV / 2; n >= 1; n >>= 1, w >>= 1) {
    const bool up = (lane & w) != 0;
#pragma unroll
    for (int i = 0; i < n; ++i) {
      const T give = up ? v[i] : v[i + n], keep = up ? v[i + n] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, give, w);
    }
  }
  T r = v[0];
  for (; w >= 1; w >>= 1) r += __shfl_xor_sync(0xffffffffu, r, w);
  return r;
}

// One warp: order |m| = blockIdx.y, degrees l0 .. l0 + NL - 1, FB fields (blockIdx.z).
template <typename T, int FB, int NL>
__global__ void __launch_bounds__(32 * kWarps) project_kernel(int L, int s, int B, const double* __restrict__ table,
                                                              const double* __restrict__ U,
                                                              const typename Cplx<T>::type* __restrict__ H,
                                                              typename Cplx<T>::type* __restrict__ flm, long long in_n,
                                                              long long out_n) {
  using C = typename Cplx<T>::type;
  constexpr int NV = 4 * NL * FB;
  static_assert(NV <= 32 && (NV & (NV - 1)) == 0, "one value a lane");
  const int Lp = L - 1, N = 2 * L - 1;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int m = blockIdx.y, b0 = blockIdx.z * FB;
  // the longest sums first
  const int l0 = m + NL * ((Lp - m) / NL - (int)(blockIdx.x * kWarps + warp));
  if (l0 < m) return;  // the whole warp
  T acc[NV];  // ((degree, field), sign, part)
#pragma unroll
  for (int k = 0; k < NV; ++k) acc[k] = T(0);
  const int last = min(l0 + NL - 1, Lp);
  for (int mp = lane; mp <= last; mp += 32) {
    T t[NL];
#pragma unroll
    for (int i = 0; i < NL; ++i) {
      const int l = l0 + i;
      t[i] = T(0);
      if (l <= last && mp <= l) t[i] = ud<T>(__ldg(&U[tri_ll(l) + mp]), __ldg(&table[doff(l) + (size_t)m * (l + 1) + mp]));
    }
#pragma unroll
    for (int j = 0; j < FB; ++j) {
      C hp, hn;
      hp.x = hp.y = hn.x = hn.y = T(0);
      if (b0 + j < B) {
        const long long ip = ((long long)(b0 + j) * N + (Lp + m)) * L + mp, in = ip - 2ll * m * L;
        if (in_bounds(ip, in_n, kbSimtIn)) hp = H[ip];
        if (in_bounds(in, in_n, kbSimtIn)) hn = H[in];
      }
#pragma unroll
      for (int i = 0; i < NL; ++i) {
        T* a = acc + 4 * (i * FB + j);
        a[0] = fma(t[i], hp.x, a[0]);
        a[1] = fma(t[i], hp.y, a[1]);
        a[2] = fma(t[i], hn.x, a[2]);
        a[3] = fma(t[i], hn.y, a[3]);
      }
    }
  }
  // the (-1)^{m'} of the +m sums follows the lane parity (m' = lane mod 32 is even/odd with lane)
  if (lane & 1) {
#pragma unroll
    for (int k = 0; k < NV; k += 4) {
      acc[k] = -acc[k];
      acc[k + 1] = -acc[k + 1];
    }
  }
  const T mine = warp_sums<T, NV>(acc, lane);
  constexpr int REP = 32 / NV;  // lanes that hold the same value
  const T other = __shfl_xor_sync(0xffffffffu, mine, REP);
  const int idx = lane / REP;
  if (lane % REP || (idx & 1)) return;  // one lane a value, the real part's lane writes
  const int sgn = (idx >> 1) & 1, q = idx >> 2, l = l0 + q / FB, b = b0 + q % FB;
  if (l > last || b >= B || (sgn && m == 0)) return;
  const int mm = sgn ? -m : m;
  // +m: (-1)^m; -m: (-1)^{l+m}
  const C out = times_ik<C>(s, sgn ? l + m : m, mm + s, mine, other);
  const long long o = (long long)b * L * L + (long long)l * l + l + mm;
  if (in_bounds(o, out_n, kbSimtOut)) flm[o] = out;
}

}  // namespace

template <typename T, int FB>
static void launch_inverse(const Dims& d, int s, int B, const double* table, const double* U, const void* flm, size_t flm_bytes,
                           void* E, size_t e_bytes, cudaStream_t st) {
  using C = typename Cplx<T>::type;
  const dim3 grid((d.L + 31) / 32, d.L, (B + FB - 1) / FB);
  inverse_kernel<T, FB><<<grid, 32 * kWarps, 0, st>>>(d.L, s, B, table, U, (const C*)flm, (C*)E,
                                                      (long long)(flm_bytes / sizeof(C)), (long long)(e_bytes / sizeof(C)));
}

template <typename T, int FB, int NL>
static void launch_project(const Dims& d, int s, int B, const double* table, const double* U, const void* H, size_t h_bytes,
                           void* flm, size_t flm_bytes, cudaStream_t st) {
  using C = typename Cplx<T>::type;
  const dim3 grid(((d.L + NL - 1) / NL + kWarps - 1) / kWarps, d.L, (B + FB - 1) / FB);
  project_kernel<T, FB, NL><<<grid, 32 * kWarps, 0, st>>>(d.L, s, B, table, U, (const C*)H, (C*)flm,
                                                          (long long)(h_bytes / sizeof(C)), (long long)(flm_bytes / sizeof(C)));
}

// Fields a thread: as many as there are, up to 4 (FP64) or 8 (FP32), in powers of two; they share the
// products U Delta and the loads of the table (a field is 4 of 5 FP64 instructions alone, 16 of 17 at 4).
template <typename T>
cudaError_t contract_inverse_simt(const Dims& d, int s, int B, const double* table, const double* U,
                                  const void* flm, size_t flm_bytes, void* E, size_t e_bytes, cudaStream_t st) {
  if (B == 1) launch_inverse<T, 1>(d, s, B, table, U, flm, flm_bytes, E, e_bytes, st);
  else if (B == 2) launch_inverse<T, 2>(d, s, B, table, U, flm, flm_bytes, E, e_bytes, st);
  else if (sizeof(T) == 8 || B <= 4) launch_inverse<T, 4>(d, s, B, table, U, flm, flm_bytes, E, e_bytes, st);
  else launch_inverse<T, sizeof(T) == 8 ? 4 : 8>(d, s, B, table, U, flm, flm_bytes, E, e_bytes, st);
  return cudaGetLastError();
}

// Degrees a warp: FP64 four with one field, two with two, one beyond, whose sums fill the lanes; FP32, which has more
// room in its pipe than in its loads of the table, two up to four fields and one beyond.  GB300, FP32, one field, by 1, 2, 4
// and 8 degrees, us: L = 256 29, 25, 29, 46; L = 1024 1394, 1133, 1539, 2949; L = 2048 10227, 8372, 11295, 21927; two fields
// by 1, 2 and 4: L = 256 35, 33, 39; L = 1024 2012, 1686, 2103.
template <typename T>
cudaError_t contract_project_simt(const Dims& d, int s, int B, const double* table, const double* U,
                                  const void* H, size_t h_bytes, void* flm, size_t flm_bytes, cudaStream_t st) {
  constexpr bool f64 = sizeof(T) == 8;
  if (B == 1) launch_project<T, 1, f64 ? 4 : 2>(d, s, B, table, U, H, h_bytes, flm, flm_bytes, st);
  else if (B == 2) launch_project<T, 2, 2>(d, s, B, table, U, H, h_bytes, flm, flm_bytes, st);
  else if (f64 || B <= 4) launch_project<T, 4, f64 ? 1 : 2>(d, s, B, table, U, H, h_bytes, flm, flm_bytes, st);
  else launch_project<T, f64 ? 4 : 8, 1>(d, s, B, table, U, H, h_bytes, flm, flm_bytes, st);
  return cudaGetLastError();
}

template cudaError_t contract_inverse_simt<double>(const Dims&, int, int, const double*, const double*, const void*, size_t, void*,
                                                   size_t, cudaStream_t);
template cudaError_t contract_inverse_simt<float>(const Dims&, int, int, const double*, const double*, const void*, size_t, void*,
                                                  size_t, cudaStream_t);
template cudaError_t contract_project_simt<double>(const Dims&, int, int, const double*, const double*, const void*, size_t, void*,
                                                   size_t, cudaStream_t);
template cudaError_t contract_project_simt<float>(const Dims&, int, int, const double*, const double*, const void*, size_t, void*,
                                                  size_t, cudaStream_t);

SSHT_BOUNDS_TU(contract_simt)

}  // namespace ssht
