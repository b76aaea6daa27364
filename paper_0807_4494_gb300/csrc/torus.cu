// The kernel between the FFTs of the triangular forward (Sec. 3.2 of the paper).
//
// Index maps.  A frequency m in [-Lp, Lp] sits at DFT bin k = m mod N; torus rows are
// stored centred (row m + Lp).  Sample theta_t = pi(2t+1)/N, so
//   sum_{m'} X_{m'} e^{i m' theta_t} = sum_k [X_{m'(k)} e^{i pi m'/N}] e^{2 pi i k t / N},
// which is how the phases of eqns dft_phase / idft_spatial enter; phi is the same.
// Phases come from a table ph[k + N - 1] = e^{i pi k / N}, |k| <= N - 1, built in FP64.
#include "ssht_internal.h"

namespace ssht {
namespace {

constexpr int TILE = 32;

// X[b][t][k] (t < L) -> ext[b][m+Lp][t'] for t' < N.
// t' < L: X[t'][k(m)] e^{-i pi m/N}/N, except t' = Lp with odd m+s -> 0; t' >= L: (-1)^{m+s} X[N-1-t'][k(m)] e^{-i pi m/N}/N.
__global__ void fwd_phi_to_theta_kernel(int L, int s, const double2* __restrict__ X, double2* __restrict__ ext,
                                        const double2* __restrict__ ph) {
  using C = double2;
  __shared__ C tile[TILE][TILE + 1];
  const int Lp = L - 1, N = 2 * L - 1;
  const int b = blockIdx.z;
  const int mi0 = blockIdx.x * TILE, tp0 = blockIdx.y * TILE;
  const C* Xb = X + (size_t)b * L * N;
  C* eb = ext + (size_t)b * N * N;
  // load: rows t' of the output tile map to source rows tsrc; columns are k(m) for the mi tile
  for (int r = threadIdx.y; r < TILE; r += blockDim.y) {
    const int tp = tp0 + r, mi = mi0 + threadIdx.x;
    C v;
    v.x = 0;
    v.y = 0;
    if (tp < N && mi < N) {
      const int m = mi - Lp;
      const int k = m >= 0 ? m : m + N;
      if (tp < L) {
        v = Xb[(size_t)tp * N + k];
      } else {
        v = Xb[(size_t)(N - 1 - tp) * N + k];
      }
    }
    tile[r][threadIdx.x] = v;
  }
  __syncthreads();
  const double inv_n = 1.0 / N;
  for (int r = threadIdx.y; r < TILE; r += blockDim.y) {
    const int mi = mi0 + r, tp = tp0 + threadIdx.x;
    if (mi < N && tp < N) {
      const int m = mi - Lp;
      const bool odd = ((m + s) & 1) != 0;
      double scale = inv_n;
      if (tp >= L && odd) scale = -scale;
      if (tp == Lp && odd) scale = 0.0;
      const C a = tile[threadIdx.x][r], w = ph[-m + N - 1];
      eb[(size_t)mi * N + tp] = make_double2((a.x * w.x - a.y * w.y) * scale, (a.x * w.y + a.y * w.x) * scale);
    }
  }
}

}  // namespace

cudaError_t fwd_phi_to_theta(const Dims& d, int s, int B, const void* X, void* ext, const double2* ph, cudaStream_t st) {
  dim3 block(TILE, 8), grid((d.N + TILE - 1) / TILE, (d.N + TILE - 1) / TILE, B);
  fwd_phi_to_theta_kernel<<<grid, block, 0, st>>>(d.L, s, (const double2*)X, (double2*)ext, ph);
  return cudaGetLastError();
}

}  // namespace ssht
