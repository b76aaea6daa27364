// Torus passes of small band-limits on CUDA cores, one launch a direction: the folded cosine and sine products of
// the torus stage (torus_gemm.cu gives the identities), theta and phi in one kernel, FP64 or FP32.
//
// All of a field's operands fit in shared memory, so a CTA takes a few fields, stages them once and walks blocks of rings
// (inverse: theta for every order at the block's rings, then phi of those rings) or of orders (analysis: phi
// for every ring at the block's orders, then theta of those orders); the blocks share no work, so that few fields
// spread over the GPU by their blocks.  A thread keeps 8 complex sums: the two signs of two orders of one parity in the
// inverse's theta, four rings or four orders elsewhere, so that what it reads serves four times.
//
// What bounds it: 16 B L^3 flops a direction on the FP64 pipe (97 % of it: L = 32, B = 1024 554 us), or in FP32 the
// shared-memory reads beside the multiply-adds (70 % of their rate: L = 16, B = 8192 38 us, L = 48, B = 512 58); a
// launch at the smallest sizes.  (Against the other forms: small_wanted.)
#include "bounds.cuh"
#include "ssht_internal.h"
#include "tc_common.cuh"
#include "torus_matrices.cuh"

#include <algorithm>

namespace ssht {
namespace {

using namespace folded;

constexpr int kThreads = 256;
constexpr int kMaxSmem = 200 * 1024;

template <typename T> struct Cplx;
template <> struct Cplx<double> { using type = double2; };
template <> struct Cplx<float> { using type = float2; };

template <typename T>
struct SmallArgs {
  using C = typename Cplx<T>::type;
  int L, s, B, nf, adjoint;  // nf: fields of a CTA
  const T* mats;
  const C* in;
  long long in_n;
  C* out;  // inverse: samples; analysis: H, or null with tiles
  long long out_n;
  TileOut to;
};

// Consecutive complex numbers from shared memory, 16 bytes at a time.
__device__ __forceinline__ void load2(const float2* p, float2 (&v)[2]) {
  const float4 a = *reinterpret_cast<const float4*>(p);
  v[0] = make_float2(a.x, a.y);
  v[1] = make_float2(a.z, a.w);
}
__device__ __forceinline__ void load2(const double2* p, double2 (&v)[2]) {
  v[0] = p[0];
  v[1] = p[1];
}
template <typename C>
__device__ __forceinline__ void load4(const C* p, C (&v)[4]) {
  C a[2];
  load2(p, a);
  v[0] = a[0];
  v[1] = a[1];
  load2(p + 2, a);
  v[2] = a[0];
  v[3] = a[1];
}
template <typename T, typename C>
__device__ __forceinline__ void axpy(C& acc, T a, C x) {
  acc.x = fma(a, x.x, acc.x);
  acc.y = fma(a, x.y, acc.y);
}
template <typename C, typename T>
__device__ __forceinline__ C cplx(T x, T y) {
  C c;
  c.x = x;
  c.y = y;
  return c;
}

// Half rows F [b][m + L - 1][m'] -> samples f [b][t][p].  blockIdx.x: fields, blockIdx.y: blocks of TB rings (every
// gridDim.y-th).
template <typename T, int TB>
__global__ void __launch_bounds__(kThreads) small_inverse_kernel(const __grid_constant__ SmallArgs<T> a) {
  using C = typename Cplx<T>::type;
  extern __shared__ __align__(16) unsigned char smem[];
  const int L = a.L, N = 2 * L - 1, ls = (L + 1) & ~1, b0 = blockIdx.x * a.nf, nf = min(a.nf, a.B - b0);
  C* const F = reinterpret_cast<C*>(smem);       // [f][m + L - 1][k], rows of ls
  C* const E = F + (size_t)a.nf * N * ls;        // [f][m][t]
  C* const O = E + a.nf * L * TB;
  T* const A = reinterpret_cast<T*>(O + a.nf * L * TB);  // cosines, sines [k][t]
  const T* const Cm = a.mats + (size_t)kCosKX * L * L;
  const T* const Sm = a.mats + (size_t)kSinKX * L * L;
  const C zero = cplx<C>(T(0), T(0));
  const long long in0 = (long long)b0 * N * L;
  for (int i = threadIdx.x; i < nf * N * ls; i += kThreads) {
    const int row = i / ls, k = i - row * ls;
    const long long at = in0 + (long long)row * L + k;
    F[i] = k < L && in_bounds(at, a.in_n, kbTorusIn) ? __ldg(&a.in[at]) : zero;
  }
  for (int t0 = blockIdx.y * TB; t0 < L; t0 += gridDim.y * TB) {
    for (int i = threadIdx.x; i < ls * TB; i += kThreads) {
      const int k = i / TB, t = t0 + i % TB;
      const bool in = k < L && t < L;
      const T half = k == 0 ? T(0.5) : T(1);  // the sums are doubled below
      A[i] = in ? half * __ldg(&Cm[k * L + t]) : T(0);
      A[ls * TB + i] = in ? half * __ldg(&Sm[k * L + t]) : T(0);
    }
    __syncthreads();
    // theta: orders m and m + 2 (one parity), both signs
    const int pairs = (L + 3) / 4 * 2;
    for (int i = threadIdx.x; i < nf * pairs * TB; i += kThreads) {
      const int t = i % TB, r = i / TB, f = r / pairs, g = r - f * pairs, m = 4 * (g >> 1) + (g & 1);
      if (m >= L) continue;
      const bool odd = (m + a.s) & 1, both = m + 2 < L;
      const T* A0 = A + (odd ? ls * TB : 0) + t;
      const C* x0 = F + (size_t)(f * N + L - 1) * ls;
      const C* row[4] = {x0 + m * ls, x0 - m * ls, x0 + (both ? m + 2 : 0) * ls, x0 - (both ? m + 2 : 0) * ls};
      C v[4] = {zero, zero, zero, zero};
#pragma unroll 2
      for (int k = 0; k < ls; k += 2) {
        const T w0 = A0[k * TB], w1 = A0[(k + 1) * TB];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          C x[2];
          load2(row[q] + k, x);
          axpy(v[q], w0, x[0]);
          axpy(v[q], w1, x[1]);
        }
      }
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        if (q == 1 && !both) break;
        const C p = v[2 * q], n = v[2 * q + 1];
        C e = cplx<C>(T(2) * (p.x + n.x), T(2) * (p.y + n.y)), o = cplx<C>(T(2) * (p.x - n.x), T(2) * (p.y - n.y));
        if (m + 2 * q == 0) {
          e = cplx<C>(T(2) * p.x, T(2) * p.y);
          o = zero;
        }
        if (odd) {  // times i
          e = cplx<C>(-e.y, e.x);
          o = cplx<C>(-o.y, o.x);
        }
        const int at = (f * L + m + 2 * q) * TB + t;
        E[at] = e;
        O[at] = o;
      }
    }
    __syncthreads();
    // phi: four rings at one sample and its mirror image
    for (int i = threadIdx.x; i < nf * (TB / 4) * L; i += kThreads) {
      const int r = i / L, p = i - r * L, t = 4 * (r % (TB / 4)), f = r / (TB / 4);
      if (t0 + t >= L) continue;
      C e[4] = {zero, zero, zero, zero}, o[4] = {zero, zero, zero, zero};
      const C* Ep = E + f * L * TB + t;
      const C* Op = O + f * L * TB + t;
#pragma unroll 2
      for (int m = 0; m < L; ++m) {
        const T c = __ldg(&Cm[m * L + p]), sn = __ldg(&Sm[m * L + p]);
        C x[4];
        load4(Ep + m * TB, x);
#pragma unroll
        for (int q = 0; q < 4; ++q) axpy(e[q], c, x[q]);
        load4(Op + m * TB, x);
#pragma unroll
        for (int q = 0; q < 4; ++q) axpy(o[q], sn, x[q]);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (t0 + t + q >= L) break;
        const long long at = ((long long)(b0 + f) * L + t0 + t + q) * N;
        if (in_bounds(at + p, a.out_n, kbTorusOut)) a.out[at + p] = cplx<C>(e[q].x - o[q].y, e[q].y + o[q].x);
        if (p < L - 1 && in_bounds(at + N - 1 - p, a.out_n, kbTorusOut))
          a.out[at + N - 1 - p] = cplx<C>(e[q].x + o[q].y, e[q].y - o[q].x);
      }
    }
    __syncthreads();
  }
}

// The projection's data tile (order m, chunk c of 32 m') of field b: rows sign * NC / 2 + 2b + part, the negative sign
// carrying (-1)^{m'}; the warp's lanes hold K = m'.
template <bool BF>
__device__ __forceinline__ void put_tile(const TileOut& to, int b, int m, int c, int lane, float2 hp, float2 hm) {
  const int sl = b / to.Bs, half = to.NC / 2, r0 = 2 * (b - sl * to.Bs), pbytes = to.NC * 128;
  const size_t tb = (size_t)tc::kParts<BF> * pbytes;
  const long long tix = sl * (long long)(to.xslice / tb) + (long long)m * to.nC + c;
  const bool ok = in_bounds(tix, (long long)(to.xbytes / tb), kbPutTile) && in_bounds(half + r0 + 1, to.NC, kbPutTile);
  const float sgn = m == 0 ? 0.f : (lane & 1) ? -1.f : 1.f;
  hm = make_float2(sgn * hm.x, sgn * hm.y);
  float sc = 0.f;
  const float up = BF ? 1.f : tc::warp_power(fmaxf(fmaxf(fabsf(hp.x), fabsf(hp.y)), fmaxf(fabsf(hm.x), fabsf(hm.y))), &sc);
  uint8_t* tile = to.X + (size_t)tix * tb;
  tc::put_rows2<BF>(tile, pbytes, r0, lane, hp.x, hp.y, up, ok);
  tc::put_rows2<BF>(tile, pbytes, half + r0, lane, hm.x, hm.y, up, ok);
  if (!BF && ok && lane == 0) {
    to.scale[(size_t)tix * half + (r0 >> 1)] = sc;
    to.scale[(size_t)tix * half + ((half + r0) >> 1)] = sc;
  }
}

// Samples f [b][t][p] -> H [b][m + L - 1][m'] (TILES 0) or the projection's data tiles (1 split FP16, 2 split BF16).
// blockIdx.x: fields, blockIdx.y: blocks of MB orders |m| (every gridDim.y-th).
template <typename T, int MB, int TILES>
__global__ void __launch_bounds__(kThreads) small_analysis_kernel(const __grid_constant__ SmallArgs<T> a) {
  using C = typename Cplx<T>::type;
  extern __shared__ __align__(16) unsigned char smem[];
  const int L = a.L, N = 2 * L - 1, ls = (L + 1) & ~1, b0 = blockIdx.x * a.nf, nf = min(a.nf, a.B - b0);
  C* const e = reinterpret_cast<C*>(smem);  // folded samples [f][t][p], rows of ls
  C* const o = e + (size_t)a.nf * L * ls;
  C* const P = o + (size_t)a.nf * L * ls;   // [f][t][j], j: the block's orders, even ones first
  C* const Q = P + a.nf * L * MB;
  const T* const Cm = a.mats + (size_t)kCosXK * L * L;
  const T* const Sm = a.mats + (size_t)kSinXK * L * L;
  const C zero = cplx<C>(T(0), T(0));
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < nf * L * ls; i += kThreads) {
    const int row = i / ls, p = i - row * ls;
    const long long at = ((long long)b0 * L + row) * N;
    C x = zero, y = zero;
    if (p < L && in_bounds(at + p, a.in_n, kbTorusIn)) x = __ldg(&a.in[at + p]);
    if (p < L - 1 && in_bounds(at + N - 1 - p, a.in_n, kbTorusIn)) y = __ldg(&a.in[at + N - 1 - p]);
    e[i] = cplx<C>(x.x + y.x, x.y + y.y);
    o[i] = p < L - 1 ? cplx<C>(x.x - y.x, x.y - y.y) : zero;
  }
  for (int m0 = blockIdx.y * MB; m0 < L; m0 += gridDim.y * MB) {
    __syncthreads();
    // phi: four rings at one order
    const int quads = (L + 3) / 4;
    for (int i = threadIdx.x; i < nf * quads * MB; i += kThreads) {
      const int j = i % MB, r = i / MB, f = r / quads, t = 4 * (r - f * quads), m = m0 + j;
      if (m >= L) continue;
      C pv[4] = {zero, zero, zero, zero}, qv[4] = {zero, zero, zero, zero};
      int at[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) at[q] = (f * L + min(t + q, L - 1)) * ls;
      for (int p = 0; p < ls; p += 2) {
        T c[2], sn[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          c[h] = p + h < L ? __ldg(&Cm[(p + h) * L + m]) : T(0);
          sn[h] = p + h < L ? __ldg(&Sm[(p + h) * L + m]) : T(0);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          C x[2];
          load2(e + at[q] + p, x);
          axpy(pv[q], c[0], x[0]);
          axpy(pv[q], c[1], x[1]);
          load2(o + at[q] + p, x);
          axpy(qv[q], sn[0], x[0]);
          axpy(qv[q], sn[1], x[1]);
        }
      }
      const int jj = (j & 1) * (MB / 2) + (j >> 1);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (t + q >= L) break;
        P[(f * L + t + q) * MB + jj] = pv[q];
        Q[(f * L + t + q) * MB + jj] = qv[q];
      }
    }
    __syncthreads();
    // theta: a warp takes 32 m' of four orders of one parity
    const int nC = (L + 31) / 32, per = MB / 4 * nC;
    for (int w = warp; w < nf * per; w += kThreads / 32) {
      const int f = w / per, r = w - f * per, c = r % nC, g = r / nC, par = g & 1, j0 = 4 * (g >> 1);
      const int m = m0 + 2 * j0 + par, mp = 32 * c + lane;
      if (m >= L) continue;
      const bool odd = (m + a.s) & 1, live = mp < L;
      const T* W = a.mats + (size_t)(a.adjoint ? (odd ? kSinXK : kCosXK) : (odd ? kWeightO : kWeightE)) * L * L + (live ? mp : 0);
      const C* Pp = P + f * L * MB + par * (MB / 2) + j0;
      const C* Qp = Q + f * L * MB + par * (MB / 2) + j0;
      C pv[4] = {zero, zero, zero, zero}, qv[4] = {zero, zero, zero, zero};
#pragma unroll 2
      for (int t = 0; t < L; ++t) {
        const T x = __ldg(&W[t * L]);
        C z[4];
        load4(Pp + t * MB, z);
#pragma unroll
        for (int q = 0; q < 4; ++q) axpy(pv[q], x, z[q]);
        load4(Qp + t * MB, z);
#pragma unroll
        for (int q = 0; q < 4; ++q) axpy(qv[q], x, z[q]);
      }
      const T twice = !live ? T(0) : a.adjoint && mp > 0 ? T(2) : T(1);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int mq = m + 2 * q;
        if (mq >= L) break;
        C hp = cplx<C>(twice * (pv[q].x + qv[q].y), twice * (pv[q].y - qv[q].x));
        C hm = cplx<C>(twice * (pv[q].x - qv[q].y), twice * (pv[q].y + qv[q].x));
        if (odd) {  // times -i
          hp = cplx<C>(hp.y, -hp.x);
          hm = cplx<C>(hm.y, -hm.x);
        }
        if constexpr (TILES == 0) {
          const long long op = ((long long)(b0 + f) * N + L - 1 + mq) * L + mp, on = op - 2ll * mq * L;
          if (live && in_bounds(op, a.out_n, kbTorusOut)) a.out[op] = hp;
          if (live && mq > 0 && in_bounds(on, a.out_n, kbTorusOut)) a.out[on] = hm;
        } else {
          if (!live) hp = hm = zero;  // (a zero times a field's NaN is one)
          put_tile<TILES == 2>(a.to, b0 + f, mq, c, lane, hp, hm);
        }
      }
    }
  }
}

}  // namespace

struct SmallPlan {
  int L = 0, sms = 0;
  bool f64 = false;
  void* mats = nullptr;
  size_t bytes = 0;
};

// Where this form is the better one.  FP32-class plans, against the tensor-core products (which round a field up to units
// of 128 rows and 64 K), inverse and forward with a kept table in us, these and those: fp32 L = 16, B = 4096 83 + 114 and
// 401 + 366, L = 48, B = 512 130 + 189 and 163 + 176, L = 49, B = 512 183 + 218 and 167 + 195, L = 64, B = 64 46 + 54 and
// 48 + 54, B = 128 79 + 96 and 68 + 85, L = 65, B = 1 35 + 37 and 33 + 30 (its 17 quads of rings take the CTA two turns);
// tf32x3 L = 48, B = 512 93 + 99 and 113 + 113, L = 64, B = 1 29 + 29 and 33 + 31, B = 128 58 + 58 and 50 + 50.
// FP64 plans, against the two-launch products (torus_direct.cu), which spread a few fields over more of the GPU's FP64 pipes:
// L = 4, B = 1 31 and 29, B = 128 32 and 38; L = 8, B = 64 42 and 40, B = 128 48 and 64; L = 16, B = 32 66 and 51, B = 128 83 and 112;
// L = 32, B = 32 131 and 104, B = 96 219 and 211, B = 128 236 and 265, B = 8192 5432 + 6481 and 6647 + 8007.
bool small_wanted(int L, int B, bool f64) {
  return f64 ? L <= 4 || (L <= 32 && B >= 128) : L <= 48 || (L <= 64 && (long long)B * L * L * L <= (1ll << 24));
}

// Rings or orders of a block: the sizes the kernels are made for.
static int block_of(int L) { return L <= 8 ? 8 : 16; }
static size_t inverse_smem(int L, int nf, size_t real) {
  const size_t ls = (L + 1) & ~1, tb = block_of(L);
  return nf * (2 * L - 1) * ls * 2 * real + 2 * nf * L * tb * 2 * real + 2 * ls * tb * real;
}
static size_t analysis_smem(int L, int nf, size_t real) {
  const size_t ls = (L + 1) & ~1, mb = block_of(L);
  return 2 * nf * L * ls * 2 * real + 2 * nf * L * mb * 2 * real;
}

template <typename T>
static cudaError_t small_attrs() {
  const void* fns[] = {(const void*)small_inverse_kernel<T, 8>, (const void*)small_inverse_kernel<T, 16>,
                       (const void*)small_analysis_kernel<T, 8, 0>, (const void*)small_analysis_kernel<T, 16, 0>};
  for (const void* fn : fns) {
    const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}
static cudaError_t small_tile_attrs() {
  const void* fns[] = {(const void*)small_analysis_kernel<float, 8, 1>, (const void*)small_analysis_kernel<float, 16, 1>,
                       (const void*)small_analysis_kernel<float, 8, 2>, (const void*)small_analysis_kernel<float, 16, 2>};
  for (const void* fn : fns) {
    const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t small_setup(SmallPlan** out, int L, bool f64, int device) {
  *out = nullptr;
  SmallPlan* p = new SmallPlan();
  p->L = L;
  p->f64 = f64;
  cudaError_t e = cudaDeviceGetAttribute(&p->sms, cudaDevAttrMultiProcessorCount, device);
  if (e == cudaSuccess) e = f64 ? small_attrs<double>() : small_attrs<float>();
  if (e == cudaSuccess && !f64) e = small_tile_attrs();
  if (e == cudaSuccess) e = f64 ? make_matrices(L, (double**)&p->mats, &p->bytes) : make_matrices(L, (float**)&p->mats, &p->bytes);
  if (e != cudaSuccess) {
    small_destroy(p);
    return e;
  }
  *out = p;
  return cudaSuccess;
}

void small_destroy(SmallPlan* p) {
  if (!p) return;
  if (p->mats) cudaFree(p->mats);
  delete p;
}

size_t small_bytes(const SmallPlan* p) { return p ? p->bytes : 0; }

// Fields of a CTA: two rounds of theta work for its threads, but no more than leave two CTAs to every SM; the blocks of
// rings or orders go to CTAs of their own while the fields alone do not fill the GPU -- in FP64, which the pipe bounds, until
// eight CTAs an SM even out its share (L = 32, B = 512 989 -> 830 us an inverse and a forward against two).
static dim3 small_grid(const SmallPlan* p, int B, int* nf) {
  const int tb = block_of(p->L), items = (p->L + 3) / 4 * 2 * tb, blocks = (p->L + tb - 1) / tb, want = 2 * p->sms;
  *nf = std::max(1, std::min({32, 2 * kThreads / items, B / want}));
  const int gx = (B + *nf - 1) / *nf, ctas = (p->f64 ? 8 : 2) * p->sms;
  return dim3((unsigned)gx, (unsigned)std::min(blocks, (ctas + gx - 1) / gx));
}

template <typename T>
static SmallArgs<T> small_args(const SmallPlan* p, int adjoint, int s, int B, const void* in, size_t in_bytes, void* out,
                               size_t out_bytes) {
  using C = typename Cplx<T>::type;
  SmallArgs<T> a{};
  a.L = p->L;
  a.s = s;
  a.B = B;
  a.adjoint = adjoint;
  a.mats = (const T*)p->mats;
  a.in = (const C*)in;
  a.in_n = (long long)(in_bytes / sizeof(C));
  a.out = (C*)out;
  a.out_n = (long long)(out_bytes / sizeof(C));
  return a;
}

template <typename T>
static cudaError_t run_inverse(const SmallPlan* p, SmallArgs<T> a, cudaStream_t st) {
  const dim3 grid = small_grid(p, a.B, &a.nf);
  const size_t smem = inverse_smem(p->L, a.nf, sizeof(T));
  if (block_of(p->L) == 8)
    small_inverse_kernel<T, 8><<<grid, kThreads, smem, st>>>(a);
  else
    small_inverse_kernel<T, 16><<<grid, kThreads, smem, st>>>(a);
  return cudaGetLastError();
}

template <typename T, int TILES>
static cudaError_t run_analysis(const SmallPlan* p, SmallArgs<T> a, cudaStream_t st) {
  const dim3 grid = small_grid(p, a.B, &a.nf);
  const size_t smem = analysis_smem(p->L, a.nf, sizeof(T));
  if (block_of(p->L) == 8)
    small_analysis_kernel<T, 8, TILES><<<grid, kThreads, smem, st>>>(a);
  else
    small_analysis_kernel<T, 16, TILES><<<grid, kThreads, smem, st>>>(a);
  return cudaGetLastError();
}

cudaError_t small_inverse(const SmallPlan* p, int s, int B, const void* F, size_t f_bytes, void* out, size_t out_bytes,
                          cudaStream_t st) {
  return p->f64 ? run_inverse(p, small_args<double>(p, 0, s, B, F, f_bytes, out, out_bytes), st)
                : run_inverse(p, small_args<float>(p, 0, s, B, F, f_bytes, out, out_bytes), st);
}

cudaError_t small_analysis(const SmallPlan* p, int adjoint, int s, int B, const void* f, size_t f_bytes, void* H, size_t h_bytes,
                           const TileOut* tiles, cudaStream_t st) {
  if (p->f64) return run_analysis<double, 0>(p, small_args<double>(p, adjoint, s, B, f, f_bytes, H, h_bytes), st);
  SmallArgs<float> a = small_args<float>(p, adjoint, s, B, f, f_bytes, H, h_bytes);
  if (!tiles) return run_analysis<float, 0>(p, a, st);
  a.to = *tiles;
  return tiles->mode == 2 ? run_analysis<float, 2>(p, a, st) : run_analysis<float, 1>(p, a, st);
}

SSHT_BOUNDS_TU(torus_small)

}  // namespace ssht
