// Internal declarations of libssht (not part of the C ABI).
#pragma once

#include <cuda_runtime.h>
#include <cufft.h>

#include <cstddef>
#include <cstdint>
#include <string>

#include "../../include/ssht.h"

namespace ssht {

// Every kernel of the library asks for the largest shared-memory carveout of the SM's unified
// L1 / shared array.  CTAs of different kernels share an SM only under one carveout, and the
// recursion (one CTA per SM for the whole sweep) is meant to share its SMs with the kernels of
// the other stream.
template <class K>
inline cudaError_t prefer_shared(K kernel) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
}

// Device status word bits (latched by kernels, read by ssht_plan_check).
enum : int { kStatusOk = 0, kStatusBarrierTimeout = 1 };

// Sizes derived from the exclusive band-limit L.
struct Dims {
  int L;   // exclusive band-limit
  int Lp;  // L - 1, the paper's inclusive band-limit
  int N;   // 2L - 1 torus samples per axis
};

// Records the message returned by ssht_last_error() and returns code.
int set_last_error(int code, const char* msg);

// Every device allocation of the library goes through here (cudaMalloc), so that the test hook
// ssht_debug_fail_allocation can make a chosen one fail as if the device were out of memory.
cudaError_t dev_malloc(void** ptr, size_t bytes);
template <class T>
inline cudaError_t dev_malloc(T** ptr, size_t bytes) {
  return dev_malloc(reinterpret_cast<void**>(ptr), bytes);
}

inline size_t delta_offset(long long l) { return (size_t)(l * (l + 1) * (2 * l + 1) / 6); }
inline size_t tri(long long l) { return (size_t)(l * (l + 1) / 2); }

// ---------------------------------------------------------------------------
// Delta recursion (delta.cu)
// ---------------------------------------------------------------------------
// How the Delta table is made: the three-term relation in m' (delta_column.cu, the default) or
// the Risbo recursion the paper uses (delta.cu).
enum : int { kDeltaColumn = 0, kDeltaRisbo = 1 };

struct DeltaWork {
  int method = kDeltaColumn;
  double* table = nullptr;        // quadrant table, delta_offset(L) doubles
  double* slab[2] = {nullptr, nullptr};  // padded octant slabs (rows 0..L, columns -1..m+1)
  double* sqrt_tab = nullptr;     // sqrt(k), k = 0 .. 2L + 2
  unsigned int* barrier = nullptr;  // grid barrier counter
  int* status = nullptr;          // latched status word
  int blocks = 0;                 // cooperative grid size
  int sms = 0;                    // SMs of the device (column method)
  int threads = 0;
  size_t smem = 0;
  size_t bytes = 0;   // device memory held (table, slabs, tables, words)
  int4* part = nullptr;   // per step and CTA: owned rows and the CTAs waited for
  size_t bytes_part = 0;
  long long cap = 0;  // shared-memory doubles per CTA
  int2* tasks = nullptr;  // column method: (degree, column block) tasks, longest first
  int ntasks = 0;
};

cudaError_t delta_setup(DeltaWork& w, int L, int device, int method = kDeltaColumn);
void delta_free(DeltaWork& w);
// wait_ns: spin limit of the Risbo recursion's waits (the column recursion has none).
constexpr long long kDefaultWaitNs = 1000000000ll;
cudaError_t delta_run(const DeltaWork& w, int L, cudaStream_t st, long long wait_ns = kDefaultWaitNs);
// The column method's setup and launch (delta_column.cu); delta_setup / delta_run dispatch.
cudaError_t column_setup(DeltaWork& w, int L, int device);
cudaError_t column_run(const DeltaWork& w, int L, cudaStream_t st);
// Those entries of the table that the spin column of s reads (column method; synchronises the stream).
cudaError_t column_run_spin(const DeltaWork& w, int L, int s, cudaStream_t st);
// U[l][m'] = sqrt((2l+1)/4pi) Delta^l_{m',-s}, l < L, 0 <= m' <= l, at tri(l) + m'; Uf is the
// same in FP32 (rounded to nearest).
cudaError_t delta_spin_column(const double* table, int L, int s, double* U, float* Uf, cudaStream_t st);

// ---------------------------------------------------------------------------
// SIMT contractions (contract_simt.cu); T is double or float
// ---------------------------------------------------------------------------
// Inverse: the half rows F[b][m + Lp][m'], 0 <= m' < L, of F (eqn fourier_coeff), the torus passes' input.
template <typename T>
cudaError_t contract_inverse_simt(const Dims& d, int s, int B, const double* table, const double* U,
                                  const void* flm, size_t flm_bytes, void* F, size_t f_bytes, cudaStream_t st);
// Projection: flm[b][l*l+l+m] = (-1)^s i^{m+s} c_l sum_{m'>=0} Delta_{m'm} Delta_{m',-s} H[b][m+Lp][m']
template <typename T>
cudaError_t contract_project_simt(const Dims& d, int s, int B, const double* table, const double* U,
                                  const void* H, size_t h_bytes, void* flm, size_t flm_bytes, cudaStream_t st);

// The paper's triangular forward (triangular.cu), FP64: Fk = theta-DFT bins of the extended
// columns [B][N][N] (no phase, no 1/N), flm [B][L*L] double2.
cudaError_t triangular_solve(const Dims& d, int s, int B, const double* table, const double* U, const void* Fk,
                             const double2* ph, void* flm, cudaStream_t st);

// Real spin-0 fields two to a complex field (real.cu); T is double or float.  flm: [nreal][L*L]
// complex, f: [nreal][L][2L-1] real; rc, rg: the complex pairs ([ceil(nreal/2)][...]).
template <typename T> cudaError_t real_pack_coeffs(int L, int nreal, const void* flm, void* rc, cudaStream_t st);
template <typename T> cudaError_t real_pack_grid(int L, int nreal, const void* f, void* rg, cudaStream_t st);
template <typename T> cudaError_t real_unpack_grid(int L, int nreal, const void* rg, void* f, cudaStream_t st);
template <typename T> cudaError_t real_unpack_coeffs(int L, int nreal, const void* rc, void* flm, cudaStream_t st);
// Spin pairs (real.cu): c [B][L*L] spin-s coefficients -> out [B][2][L*L] (spin s, then spin -s of
// the conjugate field); in [B][2][L*L] -> c [B][L*L] (the spin-s halves).
template <typename T> cudaError_t pair_expand(int L, int s, int B, const void* c, void* out, cudaStream_t st);
template <typename T> cudaError_t pair_gather(int L, int B, const void* in, void* c, cudaStream_t st);
// Kernel attributes of the packing kernels (on the current device).
cudaError_t real_setup();

// ---------------------------------------------------------------------------
// Tensor-core contractions (contract_tc.cu), split-FP16 (SSHT_TF32X3) or split-BF16
// ---------------------------------------------------------------------------
struct TcPlan;
// The contraction's tunable shape: fields per slice (the N tile: 2 x 2 x slice real columns,
// padded to 16), pipeline depth (stages of A and data tiles in shared memory), and the order of the
// work items (inverse: 0 grouped by m, 1 longest first; forward: 0 longest first, 1 grouped by m).
struct TcConfig {
  int slice = 64;
  int stages = 4;  // a new plan takes fewer where four do not fit
  int inv_order = 0;
  int fwd_order = 0;
};
// bf16 = 0: split-FP16 (two parts, three products); bf16 = 1: split-BF16 (three parts, six products).  Any batch:
// the fields run in slices of at most 64.
cudaError_t tc_setup(TcPlan** out, int L, int s, int B, int bf16, int device);
bool tc_config_fits(const TcPlan* p, const TcConfig& c);  // within the device's shared memory
cudaError_t tc_configure(TcPlan* p, const TcConfig& c);    // reallocates the data tiles if needed
TcConfig tc_config(const TcPlan* p);
void tc_destroy(TcPlan* p);
size_t tc_bytes(const TcPlan* p);
// Pack the A operand (U_l[m'] Delta^l_{m'm} in FP32, then split) of one direction from the FP64
// table and the FP32 copy of U.
cudaError_t tc_pack_a(TcPlan* p, int forward, const double* table, const float* U, cudaStream_t st, int* launches);
// Pack the inverse's data operand V from flm (float2 [B][L*L]); the forward's and the adjoint's
// data tiles come from their theta passes (TileOut).
cudaError_t tc_pack_data(TcPlan* p, const void* src, cudaStream_t st, int* launches);
// The contraction: forward = 0 writes the half rows F (float2 [B][N][L], m' >= 0) of the inverse;
// forward = 1 writes flm (float2 [B][L*L]), large outputs by way of the workspace rows (float2 [B][N][L];
// null: always directly).  Timeouts set bit 2 of *status.
cudaError_t tc_gemm(TcPlan* p, int forward, void* out, void* rows, int* status, long long wait_ns,
                    cudaStream_t st, int* launches);
// Where the forward theta pass writes the projection's data tiles directly (in place of H and
// tc_pack_data): the tile array, its column count NC, chunks per m nC, and the split form
// (mode 1: split-FP16, 2: split-BF16; 0: no tiles, H is written).
struct TileOut {
  uint8_t* X = nullptr;
  int NC = 0, nC = 0, mode = 0;
  int Bs = 64;        // fields per slice; slice z of the fields has its tiles at X + z * xslice
  size_t xslice = 0;
  size_t xbytes = 0;  // the whole tile array (index checks)
  float* scale = nullptr;  // split-FP16: [tile][NC / 2], what undoes the power of two of a row pair
};
TileOut tc_forward_tiles(const TcPlan* p);
// Where the recursion writes the A operand itself: the forward tile array and its per-m tile
// index base.
struct ATiles {
  uint8_t* A = nullptr;
  const long long* abase = nullptr;
  long long ntiles = 0;  // tiles in A (index checks)
  int bf16 = 0;          // split-BF16 tiles (two parts) instead of FP32 values
};
ATiles tc_a_tiles(const TcPlan* p);
// The column recursion writing the A tiles of a tensor-core plan directly (no FP64 table):
// A_m[l][m'] = Uf_l[m'] Delta^l_{m'm}, rounded to FP32 and stored in the plan's tile form, by the rescaled relation whose
// tables lt holds (delta_column.cu).
struct LaneTables;
cudaError_t column_run_tiles(const DeltaWork& w, const LaneTables& lt, int L, const float* Uf, ATiles t,
                             cudaStream_t st);
// The inverse contraction's A tiles (rows m', K = l): the tile array and, per
// (m, row block i), the index from which chunk kc's tile is ibase[m * nI + i] + kc.
struct InvTiles {
  uint8_t* A = nullptr;
  const long long* ibase = nullptr;
  int nI = 0;
  int nC = 0;
  long long ntiles = 0;  // tiles in A (index checks)
  int bf16 = 0;
};
InvTiles tc_inverse_tiles(const TcPlan* p);
// Plan-time tables of the recursion with one lane per degree, which writes the inverse's tiles
// directly (delta_column.cu): coefficients a(l, m'), b(l, m'), first rows (mantissa, exponent), U
// transposed, in the triangle layout [r][l] (l >= r); its tasks (column m, chunk kc of 32 degrees).
// Plan-time tables of the tile-writing recursions: the rescaled relation's
// alpha(l, m') and p(l, m') degree-major (l(l+1)/2 + m') and in the triangle layout [m'][l], the
// first rows and U transposed (delta_column.cu).
struct LaneTables {
  double* alc = nullptr;
  float* pc = nullptr;
  double* alT = nullptr;
  float* pT = nullptr;
  double* t1m = nullptr;
  int* t1e = nullptr;
  float* ufT = nullptr;
  long long* ab2 = nullptr;  // per M: the forward tile base less the row blocks below M's own
  int2* tasks = nullptr;
  unsigned int* counter = nullptr;  // next task of the plan's own sweeps (plans of a group run side by side)
  int ntasks = 0;
  bool deep = false;   // the variant for small band-limits
  int blocks = 0;      // grid of the degree-lane recursion
  int col_blocks = 0;  // grid of the column recursion writing the forward tiles
  size_t bytes = 0;
};
// Needs the column DeltaWork of the plan (its sqrt tables) and U (FP32) on the device; synchronises.
cudaError_t lane_tables_setup(LaneTables& t, const DeltaWork& w, int L, int s, const float* Uf, int nC,
                              const long long* abase, int bf16);
void lane_tables_free(LaneTables& t);
cudaError_t column_run_inverse_tiles(const DeltaWork& w, const LaneTables& t, int L, int s, InvTiles it,
                                     cudaStream_t st);

// ---------------------------------------------------------------------------
// Fused torus passes of FP32 plans (torus_gemm.cu)
// ---------------------------------------------------------------------------
// DFTs along theta and phi with the extension, phases, sin(theta) weight convolution and folds, as
// tensor-core products.  F and H: half rows (float2) [B][N][L] (m + Lp, m' >= 0); f: samples [B][L][N].
struct TorusPlan;
cudaError_t torus_setup(TorusPlan** out, int L, int device);  // synchronises
void torus_destroy(TorusPlan* p);
size_t torus_bytes(const TorusPlan* p);
// What a plan of B fields holds for the passes: workspaces of w1 (F and H too) and w2 bytes, and how many fields a slice
// has.  All in one slice: the passes' operands lie one in each workspace; several: both in w2, torus_operand_bytes apart.
struct TorusWork {
  size_t w1 = 0, w2 = 0;
  int fields = 0;
};
TorusWork torus_work(int L, int B);
size_t torus_operand_bytes(const TorusPlan* p, int B);
// Inverse of a slice of B fields, in two steps: 0 theta (F is packed into x_work, the product goes to y_work, which may
// be F), 1 phi (from y_work to the samples out).  *_bytes: extents of the buffers from the slice on
// (the index checks of bounds-checked builds).  Timeouts of the pipeline waits set bit 2 of *status.
cudaError_t torus_inverse(const TorusPlan* p, int s, int B, const void* F, size_t f_bytes, void* x_work, void* y_work, void* out,
                          size_t out_bytes, int* status, long long wait_ns, cudaStream_t st, int* launches, int step);
// Forward (adjoint = 0: extension and sin(theta) weight) or adjoint, in two steps: 0 phi (f packed into
// x_work, the product into y_work), 1 theta (from y_work into the projection's data tiles, the slice's first field being
// field b0 there, or into H without tiles; H may be x_work).
cudaError_t torus_analysis(const TorusPlan* p, int adjoint, int s, int B, const void* f, size_t f_bytes, void* x_work, void* y_work,
                           void* H, size_t h_bytes, const TileOut* tiles, int b0, int* status, long long wait_ns, cudaStream_t st,
                           int* launches, int step);

// ---------------------------------------------------------------------------
// Torus passes of FP64 plans (torus_digits.cu, torus_direct.cu) and of small band-limits (torus_small.cu)
// ---------------------------------------------------------------------------
// The same folded products as the FP32 plans' passes, on tensor cores with both operands in fixed-point digits,
// or, with little work, in FP64 on CUDA cores.  F, H: half rows (double2) [B][m + L - 1][m']; E, O: [2][B][m][t];
// P, Q: [2][B][t][m]; samples [B][t][p].
struct DigitPlan;
cudaError_t digits_setup(DigitPlan** out, int L, int device);  // synchronises
void digits_destroy(DigitPlan* p);
size_t digits_bytes(const DigitPlan* p);
size_t digits_workspace_bytes(int L, int s, int B);
// One pass: 0 theta of the inverse, F -> E, O; 1 its phi, E, O -> samples, by way of mid (E, O's size); 2 phi of forward
// and adjoint, samples -> P, Q; 3 theta of the forward (with the extension and the sin(theta) weight), 4 of the adjoint, P, Q -> H.
cudaError_t digits_pass(const DigitPlan* p, int which, int s, int B, const void* in, size_t in_bytes, void* work,
                        size_t work_bytes, void* mid, size_t mid_bytes, void* out, size_t out_bytes, int* status, long long wait_ns, cudaStream_t st);

// Small band-limits, FP64 and FP32-class plans (torus_small.cu): theta and phi in one launch on CUDA cores, no workspace.
struct SmallPlan;
bool small_wanted(int L, int B, bool f64);  // whether a plan takes this form
cudaError_t small_setup(SmallPlan** out, int L, bool f64, int device);  // synchronises
void small_destroy(SmallPlan* p);
size_t small_bytes(const SmallPlan* p);
cudaError_t small_inverse(const SmallPlan* p, int s, int B, const void* F, size_t f_bytes, void* out, size_t out_bytes,
                          cudaStream_t st);
// Samples -> H, or the projection's data tiles (FP32-class tensor-core plans).
cudaError_t small_analysis(const SmallPlan* p, int adjoint, int s, int B, const void* f, size_t f_bytes, void* H, size_t h_bytes,
                           const TileOut* tiles, cudaStream_t st);

struct DirectPlan;
bool direct_wanted(int L, int B);  // whether a plan of this band-limit and batch takes the CUDA cores
cudaError_t direct_setup(DirectPlan** out, int L);  // synchronises
void direct_destroy(DirectPlan* p);
size_t direct_bytes(const DirectPlan* p);
// step 0: theta (F -> E, O), 1: phi (E, O -> samples).
cudaError_t direct_inverse(const DirectPlan* p, int s, int B, const void* in, size_t in_bytes, void* out, size_t out_bytes,
                           cudaStream_t st, int step);
// step 0: phi (samples -> P, Q), 1: theta (P, Q -> H; adjoint = 0 with the extension and the sin(theta) weight).
cudaError_t direct_analysis(const DirectPlan* p, int adjoint, int s, int B, const void* in, size_t in_bytes, void* out,
                            size_t out_bytes, cudaStream_t st, int step);

// The contractions of FP64 plans on tensor cores (contract_digits.cu): the same results as
// contract_inverse_simt (forward = 0) and contract_project_simt, with a workspace for the data columns.
bool contract_digits_wanted(int L, int B);
size_t contract_digits_bytes(int L, int B);
cudaError_t contract_digits_setup();
cudaError_t contract_digits(int forward, int L, int s, int B, int sms, const double* table, const double* U, const void* in,
                            size_t in_bytes, void* work, size_t work_bytes, void* out, size_t out_bytes, int* status,
                            long long wait_ns, cudaStream_t st);

// ---------------------------------------------------------------------------
// Torus kernels (torus.cu)
// ---------------------------------------------------------------------------
// X[b][t][k] (phi-DFT of the samples) -> ext[b][m+Lp][t'] (theta-DFT input): the per-m parity extension, factor
// e^{-i pi m/N}/N, with the phase table ph[k + N - 1] = e^{i pi k/N}, |k| < N.
cudaError_t fwd_phi_to_theta(const Dims& d, int s, int B, const void* X, void* ext, const double2* ph, cudaStream_t st);

// ---------------------------------------------------------------------------
// Index checks of bounds-checked builds (bounds.cuh): each translation unit's record, copied out
// and cleared.
// ---------------------------------------------------------------------------
struct BoundsRecord;
cudaError_t bounds_take_torus_pass(BoundsRecord* r);
cudaError_t bounds_take_contract_tc(BoundsRecord* r);
cudaError_t bounds_take_delta_column(BoundsRecord* r);
cudaError_t bounds_take_torus_digits(BoundsRecord* r);
cudaError_t bounds_take_torus_small(BoundsRecord* r);
cudaError_t bounds_take_torus_direct(BoundsRecord* r);
cudaError_t bounds_take_contract_digits(BoundsRecord* r);
cudaError_t bounds_take_real(BoundsRecord* r);
cudaError_t bounds_take_contract_simt(BoundsRecord* r);

}  // namespace ssht
