// Plan-time tables of the torus passes' matrices, shared by the products of every form (torus_gemm.cu,
// torus_digits.cu, torus_direct.cu, torus_small.cu): cos and sin of the multiples of pi/N and the sin(theta)
// weight's matrices.
#pragma once

namespace ssht {
namespace {

// cs[r] = (cos, sin)(pi r / N), r < 2N
static __global__ void node_table_kernel(int N, double2* cs) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r < 2 * N) cs[r] = make_double2(cospi((double)r / N), sinpi((double)r / N));
}

// Prefix sums over even p = 2q >= 0 of w_e(p) e^{ip x_t}, w_e(p) = 2/(1-p^2): T[q * L + t], q < L.  A block is a warp,
// whose lanes make the weights of 32 q's at a time (a division by every thread at every step took 0.47 ms at L = 1024).
static __global__ void weight_prefix_kernel(int L, const double2* __restrict__ cs, double2* __restrict__ T) {
  const int t = blockIdx.x * 32 + threadIdx.x, N = 2 * L - 1;
  double2 sum = make_double2(0.0, 0.0);
  const int step = t < L ? (int)((2ll * (2 * t + 1)) % (2 * N)) : 0;
  int r = 0;
  for (int q0 = 0; q0 < L; q0 += 32) {
    const double p = 2.0 * (q0 + (int)threadIdx.x), mine = 2.0 / (1.0 - p * p);
    for (int i = 0; i < min(32, L - q0); ++i) {
      const double w = __shfl_sync(0xffffffffu, mine, i);
      const double2 e = cs[r];
      sum.x += w * e.x;
      sum.y += w * e.y;
      if (t < L) T[(size_t)(q0 + i) * L + t] = sum;
      r += step;
      if (r >= 2 * N) r -= 2 * N;
    }
  }
}

// Entry (m', t) of a weight matrix (parity even or odd).  With the extension about theta = pi (ring
// t = L-1 once, and zero for the odd parity) the DFT of column t is F_{m''} = c_t cos(m'' x_t) / N or
// -i c_t sin(m'' x_t) / N, and H_{m'} = (2 - delta_{m'0}) 2 pi sum_{|m''| < L} F_{m''} w_e(m'' - m').  The sum is
// e^{im' x} sum_p w_e(p) e^{ip x} over -(L-1) - m' <= p <= L-1 - m': prefix sums of both signs of p.  The
// phi pass's 1/N rides along; the odd parity's factor -i does not.
__device__ __forceinline__ double weight_entry(bool even, int L, const double2* cs, const double2* T, int mp, int t) {
  const int N = 2 * L - 1;
  if (!even && (t == L - 1 || mp == 0)) return 0.0;
  const double2 up = T[(size_t)((L - 1 - mp) / 2) * L + t], dn = T[(size_t)((L - 1 + mp) / 2) * L + t];
  const double sr = up.x + dn.x - 2.0, si = up.y - dn.y;  // sum over p of w_e(p) e^{ipx}; w_e(0) = 2 counted once
  const double2 e = cs[(int)(((long long)mp * (2 * t + 1)) % (2 * N))];
  const double c = (mp == 0 ? 1.0 : 2.0) * 6.283185307179586476925 * (t == L - 1 ? 1.0 : 2.0) / ((double)N * N);
  return c * (even ? e.x * sr - e.y * si : e.x * si + e.y * sr);
}

// The folded products' matrices for CUDA cores, each L x L, [k][row], in the element type: order k at node row,
// order row at node k, and the weight's.  sin vanishes at the node theta = pi.
namespace folded {
enum Matrix { kCosKX = 0, kSinKX, kCosXK, kSinXK, kWeightE, kWeightO, kMatrices };

template <typename T>
__global__ void matrices_kernel(int L, const double2* __restrict__ cs, const double2* __restrict__ tab, T* __restrict__ out) {
  const int N = 2 * L - 1;
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (long long)L * L) return;
  const int k = (int)(e / L), r = (int)(e % L);
  const size_t n = (size_t)L * L;
  const double2 a = cs[(int)(((long long)k * (2 * r + 1)) % (2 * N))], b = cs[(int)(((long long)r * (2 * k + 1)) % (2 * N))];
  out[kCosKX * n + e] = (T)a.x;
  out[kSinKX * n + e] = r == L - 1 ? T(0) : (T)a.y;
  out[kCosXK * n + e] = (T)b.x;
  out[kSinXK * n + e] = k == L - 1 ? T(0) : (T)b.y;
  out[kWeightE * n + e] = (T)weight_entry(true, L, cs, tab, r, k);
  out[kWeightO * n + e] = (T)weight_entry(false, L, cs, tab, r, k);
}

// Allocates and fills them; synchronises.
template <typename T>
cudaError_t make_matrices(int L, T** mats, size_t* bytes) {
  const size_t n = (size_t)L * L, ncs = 2 * (size_t)(2 * L - 1);
  double2* tmp = nullptr;
  cudaError_t e = dev_malloc(mats, kMatrices * n * sizeof(T));
  if (e != cudaSuccess) return e;
  *bytes = kMatrices * n * sizeof(T);
  e = dev_malloc(&tmp, (ncs + n) * sizeof(double2));
  if (e == cudaSuccess) {
    node_table_kernel<<<(unsigned)((ncs + 255) / 256), 256>>>(2 * L - 1, tmp);
    weight_prefix_kernel<<<(unsigned)((L + 31) / 32), 32>>>(L, tmp, tmp + ncs);
    matrices_kernel<T><<<(unsigned)((n + 255) / 256), 256>>>(L, tmp, tmp + ncs, *mats);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
  }
  if (tmp) cudaFree(tmp);
  return e;
}
}  // namespace folded

}  // namespace
}  // namespace ssht
