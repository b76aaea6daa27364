// C ABI of libssht (declared in include/ssht.h): plans, workspaces, the order of the
// stages of each transform, host-pointer staging and error reporting.
#include "ssht_internal.h"
#include "bounds.cuh"

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <string>
#include <vector>

using namespace ssht;

namespace {

thread_local std::string g_last_error;

int fail(int code, const std::string& msg) {
  g_last_error = msg;
  return code;
}

}  // namespace

namespace ssht {
int set_last_error(int code, const char* msg) { return fail(code, msg); }

namespace {
std::atomic<long long> g_alloc_countdown{0};
}

cudaError_t dev_malloc(void** ptr, size_t bytes) {
  long long n = g_alloc_countdown.load();
  while (n > 0 && !g_alloc_countdown.compare_exchange_weak(n, n - 1)) {
  }
  if (n == 1) {  // this is the chosen allocation: fail it like an exhausted device
    *ptr = nullptr;
    return cudaErrorMemoryAllocation;
  }
  return cudaMalloc(ptr, bytes);
}
}  // namespace ssht

namespace {

const char* cufft_name(cufftResult r) {
  switch (r) {
    case CUFFT_SUCCESS: return "CUFFT_SUCCESS";
    case CUFFT_INVALID_PLAN: return "CUFFT_INVALID_PLAN";
    case CUFFT_ALLOC_FAILED: return "CUFFT_ALLOC_FAILED";
    case CUFFT_INVALID_VALUE: return "CUFFT_INVALID_VALUE";
    case CUFFT_INTERNAL_ERROR: return "CUFFT_INTERNAL_ERROR";
    case CUFFT_EXEC_FAILED: return "CUFFT_EXEC_FAILED";
    case CUFFT_SETUP_FAILED: return "CUFFT_SETUP_FAILED";
    case CUFFT_INVALID_SIZE: return "CUFFT_INVALID_SIZE";
    default: return "cuFFT error";
  }
}

#define SSHT_CUDA(x, what)                                                                         \
  do {                                                                                             \
    cudaError_t e_ = (x);                                                                          \
    if (e_ != cudaSuccess) {                                                                       \
      return fail(e_ == cudaErrorMemoryAllocation ? SSHT_ENOMEM : SSHT_ECUDA,                      \
                  std::string(what) + ": " + cudaGetErrorString(e_));                              \
    }                                                                                              \
  } while (0)

#define SSHT_FFT(x, what)                                                                          \
  do {                                                                                             \
    cufftResult r_ = (x);                                                                          \
    if (r_ != CUFFT_SUCCESS) {                                                                     \
      return fail(r_ == CUFFT_ALLOC_FAILED ? SSHT_ENOMEM : SSHT_ECUDA,                             \
                  std::string(what) + ": " + cufft_name(r_));                                      \
    }                                                                                              \
  } while (0)

bool is_device_pointer(const void* p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

}  // namespace

struct ssht_plan_s {
  int device = 0;
  Dims d{};
  int s = 0, B = 0, precision = 0, delta_mode = 0;
  bool f64 = true;
  size_t elem = 16;  // bytes per complex element of the I/O and workspaces
  DeltaWork delta;
  double* U = nullptr;
  float* Uf = nullptr;  // U in FP32 (tensor-core operand packing)
  void* W1 = nullptr;
  void* W2 = nullptr;
  size_t w_bytes = 0;  // of W1 (FP64 plans: of W2 too)
  void* W3 = nullptr;
  size_t w3_bytes = 0;
  double2* ph64 = nullptr;  // phase table (the triangular forward's)
  cufftHandle fft_phi = 0, fft_theta = 0;
  bool have_phi = false, have_theta = false;
  void* stage_in = nullptr;
  size_t stage_in_bytes = 0;
  void* stage_out = nullptr;
  size_t stage_out_bytes = 0;
  bool delta_ready = false;
  bool u_fixed = false;  // U / Uf made once at creation (plans whose recursion writes the A tiles)
  long long wait_ns = kDefaultWaitNs;  // spin limit of the device-side waits
  LaneTables lane;  // tables of the recursion that writes the inverse's A tiles
  size_t bytes = 0;
  TcPlan* tc = nullptr;    // tensor-core contraction (precisions SSHT_TF32X3, SSHT_BF16X6)
  TorusPlan* torus = nullptr;  // torus products of FP32-class plans
  int torus_fields = 0;        // fields of a slice of theirs
  DigitPlan* digits = nullptr;   // torus products of FP64 plans
  DirectPlan* direct = nullptr;  // ... and of those with little work
  SmallPlan* small = nullptr;    // torus products of small band-limits, any precision
  bool contract_digits = false;  // FP64 contractions on tensor cores
  int sms = 0;                   // of the plan's device
  // The Delta recursion (and the A packing) of a call runs on a second stream, forked from the
  // caller's stream at the start of the call and joined before the contraction, so that the
  // Delta-independent work of the call (the torus stage of forward/adjoint, data packing) runs
  // beside it.
  cudaStream_t aux = nullptr;
  cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
  bool join_pending = false;
  // A plan of a group shares the Delta table of its band-limit with the group's other plans:
  // the group runs the recursion (recorded by delta_event), the plan only its spin column.
  bool delta_shared = false;
  cudaEvent_t delta_event = nullptr;
  // What the next call's recursion and packing (on aux) must wait for, instead of the whole of
  // the previous calls: ev_free after the last kernel on a caller's stream that read the Delta
  // table or U (SIMT contractions, the triangular solve, the table copy; the tensor-core path reads
  // them only on aux, in order), and ev_free_a[dir] after the tensor-core contraction that read the
  // A tiles of that direction.  Each is usable only within the capture sequence it was recorded in
  // (0 = not capturing); otherwise, or before the first record, the call forks from the caller's
  // stream as a whole.
  cudaEvent_t ev_free = nullptr;
  bool free_valid = false;
  unsigned long long free_capture = 0;
  cudaEvent_t ev_free_a[2] = {nullptr, nullptr};
  bool afree_valid[2] = {false, false};
  unsigned long long afree_capture[2] = {0, 0};
  // profiling: events bracketing each stage, folded into per-stage totals on read
  struct Ev {
    int stage;
    int lane;  // 0: the call's stream, 1: the plan's second stream
    cudaEvent_t a, b;
  };
  bool prof = false;
  std::vector<Ev> evs;
  double prof_ms[SSHT_NUM_STAGES] = {};
  long long prof_n[SSHT_NUM_STAGES] = {};
  long long launches = 0;

  // Real spin-0 fields (SSHT_FLAG_REAL): nreal caller fields ride two to a complex field; B is
  // the number of complex fields the transforms see, rc / rg their coefficients and samples.
  bool real = false;
  int nreal = 0;
  void* rc = nullptr;
  void* rg = nullptr;

  // Spin pairs (SSHT_FLAG_SPIN_PAIR): coefficients [B][2][L*L], spin s then spin -s of the
  // conjugate field; rc holds the spin-s halves.
  bool pair = false;

  // bytes of the caller's buffers
  size_t coeff_bytes() const { return (size_t)(real ? nreal : B) * d.L * d.L * elem * (pair ? 2 : 1); }
  size_t grid_bytes() const { return real ? (size_t)nreal * d.L * d.N * (elem / 2) : (size_t)B * d.L * d.N * elem; }
  size_t pair_coeff_bytes() const { return (size_t)B * d.L * d.L * elem; }
  size_t pair_grid_bytes() const { return (size_t)B * d.L * d.N * elem; }
};

namespace {

void fold_events(ssht_plan_t p) {
  for (auto& e : p->evs) {
    float ms = 0.f;
    if (cudaEventSynchronize(e.b) == cudaSuccess && cudaEventElapsedTime(&ms, e.a, e.b) == cudaSuccess) {
      p->prof_ms[e.stage] += ms;
      p->prof_n[e.stage] += 1;
    }
    cudaEventDestroy(e.a);
    cudaEventDestroy(e.b);
  }
  p->evs.clear();
}

// Brackets one stage with events on the call's stream while profiling is enabled.
struct StageScope {
  ssht_plan_t p;
  int stage;
  cudaStream_t st;
  cudaEvent_t a = nullptr;
  StageScope(ssht_plan_t p_, int stage_, cudaStream_t st_) : p(p_), stage(stage_), st(st_) {
    if (p->prof && cudaEventCreate(&a) == cudaSuccess) cudaEventRecord(a, st);
  }
  ~StageScope() {
    if (!a) return;
    cudaEvent_t b;
    if (cudaEventCreate(&b) != cudaSuccess) {
      cudaEventDestroy(a);
      return;
    }
    cudaEventRecord(b, st);
    p->evs.push_back({stage, st == p->aux ? 1 : 0, a, b});
    if (p->evs.size() > 8192) fold_events(p);
  }
};

int dalloc(ssht_plan_t p, void** ptr, size_t bytes, const char* what) {
  cudaError_t e = dev_malloc(ptr, bytes ? bytes : 16);
  if (e != cudaSuccess) {
    *ptr = nullptr;
    cudaGetLastError();
    return fail(SSHT_ENOMEM, std::string("cudaMalloc ") + what + " (" + std::to_string(bytes) + " bytes): " +
                                 cudaGetErrorString(e));
  }
  p->bytes += bytes;
  return 0;
}

int run_dft(ssht_plan_t p, cufftHandle h, void* in, void* out, cudaStream_t st) {
  StageScope sc(p, SSHT_STAGE_FFT, st);
  SSHT_FFT(cufftExecZ2Z(h, (cufftDoubleComplex*)in, (cufftDoubleComplex*)out, CUFFT_FORWARD), "cufftExecZ2Z");
  return 0;
}

// The torus passes of an FP32-class plan (products along theta or phi), timed as FFT work, by slices of fields.
// Inverse: F in W1 -> samples f.
int torus_inverse_passes(ssht_plan_t p, void* f, cudaStream_t st) {
  const size_t row = (size_t)p->d.N * p->d.L * p->elem;  // of a field's half rows, and of its samples
  const bool whole = p->torus_fields == p->B;
  for (int b0 = 0; b0 < p->B; b0 += p->torus_fields) {
    const int n = std::min(p->torus_fields, p->B - b0);
    char* F = (char*)p->W1 + b0 * row;
    void* y = whole ? p->W1 : (char*)p->W2 + torus_operand_bytes(p->torus, p->torus_fields);
    for (int step = 0; step < 2; ++step) {
      StageScope sc(p, SSHT_STAGE_FFT, st);
      int k = 0;
      SSHT_CUDA(torus_inverse(p->torus, p->s, n, F, p->w_bytes - b0 * row, p->W2, y, (char*)f + b0 * row, p->pair_grid_bytes() - b0 * row,
                              p->delta.status, p->wait_ns, st, &k, step),
                "torus pass");
      p->launches += k;
    }
  }
  return 0;
}
// Forward / adjoint: samples f -> the projection's data tiles (tensor-core plans) or H in W1.
int torus_analysis_passes(ssht_plan_t p, int adjoint, const void* f, cudaStream_t st) {
  const size_t row = (size_t)p->d.N * p->d.L * p->elem;
  const bool whole = p->torus_fields == p->B;
  TileOut tiles;
  if (p->tc) tiles = tc_forward_tiles(p->tc);
  for (int b0 = 0; b0 < p->B; b0 += p->torus_fields) {
    const int n = std::min(p->torus_fields, p->B - b0);
    void* x = whole ? p->W1 : p->W2;
    void* y = whole ? p->W2 : (char*)p->W2 + torus_operand_bytes(p->torus, p->torus_fields);
    for (int step = 0; step < 2; ++step) {
      StageScope sc(p, SSHT_STAGE_FFT, st);
      int k = 0;
      SSHT_CUDA(torus_analysis(p->torus, adjoint, p->s, n, (const char*)f + b0 * row, p->pair_grid_bytes() - b0 * row, x, y,
                               (char*)p->W1 + b0 * row, p->w_bytes - b0 * row, p->tc ? &tiles : nullptr, b0, p->delta.status,
                               p->wait_ns, st, &k, step),
                "torus pass");
      p->launches += k;
    }
  }
  return 0;
}

int make_fft(ssht_plan_t p, cufftHandle* h, bool* have, int n, size_t batch, const char* what) {
  if (batch > (size_t)0x7fffffff) return fail(SSHT_EUNSUPPORTED, std::string(what) + ": batch too large");
  int nn = n;
  SSHT_FFT(cufftPlanMany(h, 1, &nn, nullptr, 1, n, nullptr, 1, n, CUFFT_Z2Z, (int)batch), what);
  *have = true;
  size_t ws = 0;
  if (cufftGetSize(*h, &ws) == CUFFT_SUCCESS) p->bytes += ws;
  return 0;
}

int set_streams(ssht_plan_t p, cudaStream_t st) {
  if (p->have_phi) SSHT_FFT(cufftSetStream(p->fft_phi, st), "cufftSetStream");
  if (p->have_theta) SSHT_FFT(cufftSetStream(p->fft_theta, st), "cufftSetStream");
  return 0;
}

int pack_a(ssht_plan_t p, int forward, cudaStream_t st);

int run_delta(ssht_plan_t p, cudaStream_t st) {
  StageScope sc(p, SSHT_STAGE_DELTA, st);
  if (!p->delta_shared) {
    SSHT_CUDA(delta_run(p->delta, p->d.L, st, p->wait_ns), "Delta recursion launch");
    p->launches += 1;
  }
  if (!p->u_fixed) {
    SSHT_CUDA(delta_spin_column(p->delta.table, p->d.L, p->s, p->U, p->Uf, st), "spin column launch");
    p->launches += 1;
  }
  return 0;
}

// Tensor-core plans with the column recursion make the contraction's A tiles in the recursion
// itself (no FP64 table, no packing): the forward's tiles (rows l, K = m') with one lane per column,
// the inverse's (rows m', K = l) with one lane per degree.  U, the spin column, and the degree-lane
// recursion's tables are made once at plan creation.  The plans of a group too, each for its own
// spin: a sweep into the tiles writes them once, while packing them from a shared FP64 table also
// reads that table (8 bytes an entry, the inverse's in columns).  Split-BF16, inverse + forward: B = 64,
// L = 1024 16.0 -> 12.5 ms, B = 16, L = 2048 62.1 -> 40.6 ms (GB300).
bool tiles_direct(const ssht_plan_s* p) { return p->tc && p->delta.method == kDeltaColumn; }

// Delta and the contraction's A operand of one direction, on st.
int make_operands(ssht_plan_t p, int forward, cudaStream_t st) {
  if (tiles_direct(p)) {
    StageScope sc(p, forward ? SSHT_STAGE_DELTA : SSHT_STAGE_DELTA_INVERSE, st);
    if (forward)
      SSHT_CUDA(column_run_tiles(p->delta, p->lane, p->d.L, p->Uf, tc_a_tiles(p->tc), st), "recursion into the A tiles");
    else
      SSHT_CUDA(column_run_inverse_tiles(p->delta, p->lane, p->d.L, p->s, tc_inverse_tiles(p->tc), st),
                "recursion into the inverse's A tiles");
    p->launches += 1;
    return 0;
  }
  int rc = run_delta(p, st);
  if (rc) return rc;
  return p->tc ? pack_a(p, forward, st) : 0;
}

int pack_a(ssht_plan_t p, int forward, cudaStream_t st) {
  StageScope sc(p, SSHT_STAGE_PACK, st);
  int n = 0;
  SSHT_CUDA(tc_pack_a(p->tc, forward, p->delta.table, p->Uf, st, &n), "tensor-core operand packing");
  p->launches += n;
  return 0;
}

int ensure_delta(ssht_plan_t p, cudaStream_t st) {
  if (p->delta_mode == SSHT_DELTA_CACHE && p->delta_ready) return 0;
  int rc = run_delta(p, st);
  if (rc) return rc;
  if (p->delta_mode == SSHT_DELTA_CACHE) p->delta_ready = true;
  return 0;
}

// Start making Delta (and, for the tensor-core path, the packed A operand of one direction) on
// the plan's second stream, after everything already queued on st; join_operands makes st wait.
unsigned long long capture_id(cudaStream_t st) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  unsigned long long id = 0;
  if (cudaStreamGetCaptureInfo(st, &cs, &id) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return cs == cudaStreamCaptureStatusActive ? id : 0;
}

// After the last reader of the table, U and the A tiles in a call.
int mark_free(ssht_plan_t p, cudaStream_t st) {
  SSHT_CUDA(cudaEventRecord(p->ev_free, st), "operands-free event");
  p->free_valid = true;
  p->free_capture = capture_id(st);
  return 0;
}

// After the tensor-core contraction of one direction: the A tiles of that direction are free.
int mark_free_a(ssht_plan_t p, int forward, cudaStream_t st) {
  SSHT_CUDA(cudaEventRecord(p->ev_free_a[forward], st), "A-tiles-free event");
  p->afree_valid[forward] = true;
  p->afree_capture[forward] = capture_id(st);
  return 0;
}

// The inverse's A tiles of a plan whose recursions write them are made as soon as the previous
// inverse contraction has read them, without waiting for the forward contraction in between: the
// degree-lane recursion (no shared memory) then fills the gaps beside the forward's packing and passes.
#ifndef SSHT_INVERSE_OPERANDS_EARLY
#define SSHT_INVERSE_OPERANDS_EARLY 1
#endif

int begin_operands(ssht_plan_t p, int forward, cudaStream_t st) {
  if (p->delta_mode == SSHT_DELTA_CACHE && p->delta_ready) return 0;
  const unsigned long long cap = capture_id(st);
  // the previous readers of what the aux work overwrites, if they are known
  const bool table_ok = !p->free_valid || p->free_capture == cap;
  const bool a_ok = !p->tc || !p->afree_valid[forward] || p->afree_capture[forward] == cap;
  const bool any = p->free_valid || (p->tc && p->afree_valid[forward]);
  if (table_ok && a_ok && any) {
    // only those readers: the rest of the previous calls (e.g. the inverse's torus stage) may
    // still be running while this call's recursion starts
    if (p->free_valid) SSHT_CUDA(cudaStreamWaitEvent(p->aux, p->ev_free, 0), "operands-free wait");
    if (p->tc && p->afree_valid[forward]) SSHT_CUDA(cudaStreamWaitEvent(p->aux, p->ev_free_a[forward], 0), "A-free wait");
    // ... and the other direction's contraction: it cannot share an SM with the recursion, so
    // queued behind a running recursion it would wait for the whole sweep, while run first
    // (about 1 ms) it lets the torus passes that follow it overlap the recursion (not for the
    // inverse's tiles of a tensor-core plan, see above)
    const bool early = SSHT_INVERSE_OPERANDS_EARLY && !forward && tiles_direct(p);
    if (p->tc && !early && p->afree_valid[1 - forward] && p->afree_capture[1 - forward] == cap)
      SSHT_CUDA(cudaStreamWaitEvent(p->aux, p->ev_free_a[1 - forward], 0), "other contraction wait");
  } else {
    SSHT_CUDA(cudaEventRecord(p->ev_fork, st), "fork event");
    SSHT_CUDA(cudaStreamWaitEvent(p->aux, p->ev_fork, 0), "fork wait");
  }
  if (p->delta_shared && p->delta_event && !tiles_direct(p)) SSHT_CUDA(cudaStreamWaitEvent(p->aux, p->delta_event, 0), "shared Delta wait");
  int rc = make_operands(p, forward, p->aux);
  if (rc) return rc;
  SSHT_CUDA(cudaEventRecord(p->ev_join, p->aux), "join event");
  p->join_pending = true;
  return 0;
}

int join_operands(ssht_plan_t p, cudaStream_t st) {
  if (!p->join_pending) return 0;
  p->join_pending = false;
  SSHT_CUDA(cudaStreamWaitEvent(st, p->ev_join, 0), "join wait");
  return 0;
}

int tc_pack(ssht_plan_t p, const void* src, cudaStream_t st) {
  int n = 0;
  StageScope sc(p, SSHT_STAGE_PACK, st);
  SSHT_CUDA(tc_pack_data(p->tc, src, st, &n), "tensor-core data packing");
  p->launches += n;
  return 0;
}

int tc_multiply(ssht_plan_t p, int forward, void* dst, cudaStream_t st) {
  int n = 0;
  StageScope sc(p, forward ? SSHT_STAGE_PROJECT : SSHT_STAGE_INVERSE, st);
  SSHT_CUDA(tc_gemm(p->tc, forward, dst, forward ? p->W1 : nullptr, p->delta.status, p->wait_ns, st, &n), "tensor-core contraction");
  p->launches += n;
  return 0;
}

// One torus product of an FP64 plan, timed as FFT work; which: 0, 1 the inverse's theta and phi, 2 phi of
// forward and adjoint, 3, 4 theta of forward and adjoint.  W1 (half rows) <-> W2 <-> samples.
int fp64_pass(ssht_plan_t p, int which, const void* in, void* out, cudaStream_t st) {
  StageScope sc(p, SSHT_STAGE_FFT, st);
  cudaError_t e;
  const size_t fb = p->pair_grid_bytes(), ib = which == 2 ? fb : p->w_bytes, ob = which == 1 ? fb : p->w_bytes;
  if (p->digits) {
    e = digits_pass(p->digits, which, p->s, p->B, in, ib, p->W3, p->w3_bytes, p->W1, p->w_bytes, out, ob, p->delta.status,
                    p->wait_ns, st);
  } else if (which < 2) {
    e = direct_inverse(p->direct, p->s, p->B, in, ib, out, ob, st, which);
  } else {
    e = direct_analysis(p->direct, which == 4, p->s, p->B, in, ib, out, ob, st, which - 2 > 0);
  }
  SSHT_CUDA(e, "torus product");
  p->launches += !p->digits ? 1 : which == 1 ? 3 : 2;
  return 0;
}

// The torus stage: half rows in W1 -> samples f.
int torus_to_samples(ssht_plan_t p, void* f, cudaStream_t st) {
  int rc;
  if (p->small) {
    StageScope sc(p, SSHT_STAGE_FFT, st);
    SSHT_CUDA(small_inverse(p->small, p->s, p->B, p->W1, p->w_bytes, f, p->pair_grid_bytes(), st), "torus product");
    p->launches += 1;
    return 0;
  }
  if (p->torus) return torus_inverse_passes(p, f, st);
  return (rc = fp64_pass(p, 0, p->W1, p->W2, st)) ? rc : fp64_pass(p, 1, p->W2, f, st);
}

// Forward / adjoint: samples f -> H in W1, or (tensor-core plans) the projection's data tiles (no H, no data
// packing).
int torus_from_samples(ssht_plan_t p, int adjoint, const void* f, cudaStream_t st) {
  int rc;
  if (p->small) {
    StageScope sc(p, SSHT_STAGE_FFT, st);
    TileOut tiles;
    if (p->tc) tiles = tc_forward_tiles(p->tc);
    SSHT_CUDA(small_analysis(p->small, adjoint, p->s, p->B, f, p->pair_grid_bytes(), p->W1, p->w_bytes, p->tc ? &tiles : nullptr, st),
              "torus product");
    p->launches += 1;
    return 0;
  }
  if (p->torus) return torus_analysis_passes(p, adjoint, f, st);
  return (rc = fp64_pass(p, 2, f, p->W2, st)) ? rc : fp64_pass(p, adjoint ? 4 : 3, p->W2, p->W1, st);
}

// The SIMT projection of forward / adjoint from the folded torus sums H (in W), after the join
// (tensor-core plans: analysis_impl).
template <typename T>
int project(ssht_plan_t p, const void* H, void* flm, cudaStream_t st) {
  int rc;
  if ((rc = join_operands(p, st))) return rc;
  {
    StageScope sc(p, SSHT_STAGE_PROJECT, st);
    if (p->contract_digits)
      SSHT_CUDA(contract_digits(1, p->d.L, p->s, p->B, p->sms, p->delta.table, p->U, H, p->w_bytes, p->W3, p->w3_bytes, flm,
                                p->pair_coeff_bytes(), p->delta.status, p->wait_ns, st),
                "projection");
    else
      SSHT_CUDA(contract_project_simt<T>(p->d, p->s, p->B, p->delta.table, p->U, H, p->w_bytes, flm, p->pair_coeff_bytes(), st),
                "projection");
    p->launches += p->contract_digits ? 2 : 1;
  }
  return mark_free(p, st);
}

int check_device(ssht_plan_t p) {
  int cur = -1;
  SSHT_CUDA(cudaGetDevice(&cur), "cudaGetDevice");
  if (cur != p->device)
    return fail(SSHT_EINVAL, "plan was created on device " + std::to_string(p->device) + " but device " +
                                 std::to_string(cur) + " is current");
  return 0;
}

int stage_buffer(ssht_plan_t p, void** buf, size_t* have, size_t need, const char* what) {
  if (*have >= need) return 0;
  if (*buf) {
    cudaFree(*buf);
    p->bytes -= *have;
    *buf = nullptr;
    *have = 0;
  }
  int rc = dalloc(p, buf, need, what);
  if (rc) return rc;
  *have = need;
  return 0;
}

// Resolve input/output pointers: host buffers go through plan-owned staging memory.
struct IO {
  const void* in_dev;
  void* out_dev;
  void* out_host;
  size_t out_bytes;
};

// A host input is copied to plan-owned device memory by the copy engines (cudaMemcpyAsync on the
// call's stream), not read in place by the first kernel over the host link: a kernel reading host
// memory holds its SMs for the whole transfer, while the copy engines leave them to the work of
// other streams (the plan's own recursion on its second stream, or another request's kernels).
int io_begin(ssht_plan_t p, const void* in, size_t in_bytes, void* out, size_t out_bytes, cudaStream_t st, IO* io) {
  if (!in || !out) return fail(SSHT_EINVAL, "null data pointer");
  io->out_host = nullptr;
  io->out_bytes = out_bytes;
  if (is_device_pointer(in)) {
    io->in_dev = in;
  } else {
    int rc = stage_buffer(p, &p->stage_in, &p->stage_in_bytes, in_bytes, "input staging");
    if (rc) return rc;
    SSHT_CUDA(cudaMemcpyAsync(p->stage_in, in, in_bytes, cudaMemcpyHostToDevice, st), "input copy to device");
    io->in_dev = p->stage_in;
  }
  if (is_device_pointer(out)) {
    io->out_dev = out;
  } else {
    int rc = stage_buffer(p, &p->stage_out, &p->stage_out_bytes, out_bytes, "output staging");
    if (rc) return rc;
    io->out_dev = p->stage_out;
    io->out_host = out;
  }
  return 0;
}

int io_end(ssht_plan_t p, const IO& io, cudaStream_t st) {
  (void)p;
  if (io.out_host) {
    SSHT_CUDA(cudaMemcpyAsync(io.out_host, io.out_dev, io.out_bytes, cudaMemcpyDeviceToHost, st),
              "output copy to host");
    SSHT_CUDA(cudaStreamSynchronize(st), "stream synchronize");
  }
  SSHT_CUDA(cudaGetLastError(), "kernel launch");
  return 0;
}

template <typename T>
int inverse_impl(ssht_plan_t p, const void* flm, void* f, cudaStream_t st) {
  const Dims& d = p->d;
  int rc = begin_operands(p, 0, st);
  if (rc) return rc;
  if (p->tc) {
    if ((rc = tc_pack(p, flm, st)) || (rc = join_operands(p, st)) || (rc = tc_multiply(p, 0, p->W1, st)) ||
        (rc = mark_free_a(p, 0, st)))
      return rc;
  } else {
    if ((rc = join_operands(p, st))) return rc;
    StageScope sc(p, SSHT_STAGE_INVERSE, st);
    if (p->contract_digits)
      SSHT_CUDA(contract_digits(0, d.L, p->s, p->B, p->sms, p->delta.table, p->U, flm, p->pair_coeff_bytes(), p->W3, p->w3_bytes,
                                p->W1, p->w_bytes, p->delta.status, p->wait_ns, st),
                "inverse contraction");
    else
      SSHT_CUDA(contract_inverse_simt<T>(d, p->s, p->B, p->delta.table, p->U, flm, p->pair_coeff_bytes(), p->W1, p->w_bytes,
                                         st),
                "inverse contraction");
    p->launches += p->contract_digits ? 2 : 1;
  }
  if (!p->tc && (rc = mark_free(p, st))) return rc;
  return torus_to_samples(p, f, st);
}

// Front of the triangular forward: phi DFT, extension into the theta-DFT input, theta DFT in place in W1.
int analysis_front(ssht_plan_t p, const void* f, cudaStream_t st) {
  const Dims& d = p->d;
  int rc = run_dft(p, p->fft_phi, const_cast<void*>(f), p->W2, st);
  if (rc) return rc;
  {
    StageScope sc(p, SSHT_STAGE_TORUS, st);
    SSHT_CUDA(fwd_phi_to_theta(d, p->s, p->B, p->W2, p->W1, p->ph64, st), "phi-to-theta extension");
    p->launches += 1;
  }
  return run_dft(p, p->fft_theta, p->W1, p->W1, st);
}

// Forward, or (adjoint) the adjoint.
template <typename T>
int analysis_impl(ssht_plan_t p, int adjoint, const void* f, void* flm, cudaStream_t st) {
  int rc = begin_operands(p, 1, st);
  if (rc || (rc = torus_from_samples(p, adjoint, f, st))) return rc;
  if (!p->tc) return project<T>(p, p->W1, flm, st);
  if ((rc = join_operands(p, st)) || (rc = tc_multiply(p, 1, flm, st))) return rc;
  return mark_free_a(p, 1, st);
}
template <typename T>
int forward_impl(ssht_plan_t p, const void* f, void* flm, cudaStream_t st) {
  return analysis_impl<T>(p, 0, f, flm, st);
}
template <typename T>
int adjoint_impl(ssht_plan_t p, const void* g, void* flm, cudaStream_t st) {
  return analysis_impl<T>(p, 1, g, flm, st);
}

// Real spin-0 fields, two to a complex field: which = 0 inverse, 1 forward, 2 adjoint.
template <typename T>
int real_call(ssht_plan_t p, int which, const void* in, void* out, cudaStream_t st) {
  const int L = p->d.L;
  int rc;
  {
    StageScope sc(p, SSHT_STAGE_PACK, st);
    if (which == 0) SSHT_CUDA(real_pack_coeffs<T>(L, p->nreal, in, p->rc, st), "real-field packing");
    else SSHT_CUDA(real_pack_grid<T>(L, p->nreal, in, p->rg, st), "real-field packing");
    p->launches += 1;
  }
  if (which == 0) rc = inverse_impl<T>(p, p->rc, p->rg, st);
  else if (which == 1) rc = forward_impl<T>(p, p->rg, p->rc, st);
  else rc = adjoint_impl<T>(p, p->rg, p->rc, st);
  if (rc) return rc;
  StageScope sc(p, SSHT_STAGE_PACK, st);
  if (which == 0) SSHT_CUDA(real_unpack_grid<T>(L, p->nreal, p->rg, out, st), "real-field unpacking");
  else SSHT_CUDA(real_unpack_coeffs<T>(L, p->nreal, p->rc, out, st), "real-field unpacking");
  p->launches += 1;
  return 0;
}

// Spin pairs: which = 0 inverse (from the spin-s halves), 1 forward, 2 adjoint (one spin-s
// transform, then the spin -s coefficients of the conjugate field by the conjugate symmetry).
template <typename T>
int pair_call(ssht_plan_t p, int which, const void* in, void* out, cudaStream_t st) {
  const int L = p->d.L;
  int rc;
  if (which == 0) {
    {
      StageScope sc(p, SSHT_STAGE_PACK, st);
      SSHT_CUDA(pair_gather<T>(L, p->B, in, p->rc, st), "spin-pair gather");
      p->launches += 1;
    }
    return inverse_impl<T>(p, p->rc, out, st);
  }
  rc = which == 1 ? forward_impl<T>(p, in, p->rc, st) : adjoint_impl<T>(p, in, p->rc, st);
  if (rc) return rc;
  StageScope sc(p, SSHT_STAGE_PACK, st);
  SSHT_CUDA(pair_expand<T>(L, p->s, p->B, p->rc, out, st), "spin-pair expansion");
  p->launches += 1;
  return 0;
}

// ---------------------------------------------------------------------------------------------
// Tile tuning of the tensor-core contraction (SSHT_FLAG_TUNE, and the tuned buckets of groups):
// every shape candidate -- fields per slice, pipeline depth, work order -- is timed on the
// plan's own operands (inverse + forward contractions, CUDA events) and the fastest kept.  With
// SSHT_TUNE_CACHE naming a file, choices are looked up there first and stored after tuning, one
// JSON object per line: {"key": "L=1024 s=2 B=64 tf32x3", "slice": 64, "stages": 2, ...}.
// ---------------------------------------------------------------------------------------------
std::string tune_key(const ssht_plan_s* p) {
  return "L=" + std::to_string(p->d.L) + " s=" + std::to_string(p->s) + " B=" + std::to_string(p->B) +
         (p->precision == SSHT_BF16X6 ? " bf16x6" : " tf32x3");
}

bool tune_cache_lookup(const std::string& key, TcConfig* c) {
  const char* path = std::getenv("SSHT_TUNE_CACHE");
  if (!path || !*path) return false;
  FILE* f = std::fopen(path, "r");
  if (!f) return false;
  char line[512];
  bool found = false;
  const std::string want = "{\"key\": \"" + key + "\",";
  while (std::fgets(line, sizeof line, f)) {
    if (std::strncmp(line, want.c_str(), want.size()) != 0) continue;
    TcConfig t;
    if (std::sscanf(line + want.size(), " \"slice\": %d, \"stages\": %d, \"inv_order\": %d, \"fwd_order\": %d", &t.slice,
                    &t.stages, &t.inv_order, &t.fwd_order) == 4) {
      *c = t;
      found = true;  // the last entry of a key wins
    }
  }
  std::fclose(f);
  return found;
}

void tune_cache_store(const std::string& key, const TcConfig& c, float ms) {
  const char* path = std::getenv("SSHT_TUNE_CACHE");
  if (!path || !*path) return;
  FILE* f = std::fopen(path, "a");
  if (!f) return;
  std::fprintf(f, "{\"key\": \"%s\", \"slice\": %d, \"stages\": %d, \"inv_order\": %d, \"fwd_order\": %d, \"ms\": %.4f}\n",
               key.c_str(), c.slice, c.stages, c.inv_order, c.fwd_order, ms);
  std::fclose(f);
}

int make_operands(ssht_plan_t p, int forward, cudaStream_t st);

// Mean milliseconds of one inverse + one forward contraction of the plan's current shape.
int time_contractions(ssht_plan_t p, cudaStream_t st, float* ms) {
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  SSHT_CUDA(cudaEventCreate(&e0), "tuning event");
  SSHT_CUDA(cudaEventCreate(&e1), "tuning event");
  int n = 0, rc = 0;
  for (int it = 0; it < 4 && !rc; ++it) {
    if (it == 1) cudaEventRecord(e0, st);
    cudaError_t e = tc_gemm(p->tc, 0, p->W1, nullptr, p->delta.status, p->wait_ns, st, &n);
    if (e == cudaSuccess) e = tc_gemm(p->tc, 1, p->W2, p->W1, p->delta.status, p->wait_ns, st, &n);
    if (e != cudaSuccess) rc = fail(SSHT_ECUDA, std::string("tuning contraction: ") + cudaGetErrorString(e));
  }
  cudaEventRecord(e1, st);
  cudaEventSynchronize(e1);
  float t = 0.f;
  cudaEventElapsedTime(&t, e0, e1);
  *ms = t / 3.f;
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  return rc;
}

int tune_tiles(ssht_plan_t p) {
  if (!p->tc) return 0;
  TcConfig best = tc_config(p->tc);
  const std::string key = tune_key(p);
  if (tune_cache_lookup(key, &best) && tc_config_fits(p->tc, best)) {
    SSHT_CUDA(tc_configure(p->tc, best), "tile configuration");
    return 0;
  }
  cudaStream_t st = nullptr;
  SSHT_CUDA(cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking), "tuning stream");
  auto done = [&](int rc) {
    cudaStreamSynchronize(st);
    cudaStreamDestroy(st);
    return rc;
  };
  int rc = 0;
  // the operands of both directions, once (the data tiles' values do not change the timing)
  if ((rc = make_operands(p, 0, st)) || (rc = make_operands(p, 1, st))) return done(rc);
  float best_ms = 0.f;
  bool have = false;
  auto trial = [&](const TcConfig& c) {
    if (!tc_config_fits(p->tc, c)) return 0;
    cudaError_t e = tc_configure(p->tc, c);
    if (e != cudaSuccess) return fail(SSHT_ECUDA, std::string("tile configuration: ") + cudaGetErrorString(e));
    float ms = 0.f;
    int r = time_contractions(p, st, &ms);
    if (r) return r;
    if (!have || ms < best_ms) {
      best_ms = ms;
      best = c;
      have = true;
    }
    return 0;
  };
  std::vector<int> slices;
  for (int sl : {64, 32, 16}) {
    const int bs = std::min(sl, p->B);
    if (std::find(slices.begin(), slices.end(), bs) == slices.end()) slices.push_back(bs);
  }
  for (int sl : slices)
    for (int stg = 2; stg <= 4; ++stg) {
      TcConfig c;
      c.slice = sl;
      c.stages = stg;
      if ((rc = trial(c))) return done(rc);
    }
  const TcConfig shape = best;
  for (int io = 0; io < 2; ++io)
    for (int fo = 0; fo < 2; ++fo) {
      if (io == shape.inv_order && fo == shape.fwd_order) continue;
      TcConfig c = shape;
      c.inv_order = io;
      c.fwd_order = fo;
      if ((rc = trial(c))) return done(rc);
    }
  cudaError_t e = tc_configure(p->tc, best);
  if (e != cudaSuccess) return done(fail(SSHT_ECUDA, std::string("tile configuration: ") + cudaGetErrorString(e)));
  tune_cache_store(key, best, best_ms);
  return done(0);
}

void release(ssht_plan_t p) {
  if (!p) return;
  cudaDeviceSynchronize();
  for (auto& e : p->evs) {
    cudaEventDestroy(e.a);
    cudaEventDestroy(e.b);
  }
  if (p->tc) tc_destroy(p->tc);
  if (p->torus) torus_destroy(p->torus);
  if (p->direct) direct_destroy(p->direct);
  if (p->small) small_destroy(p->small);
  if (p->digits) digits_destroy(p->digits);
  if (p->ev_fork) cudaEventDestroy(p->ev_fork);
  if (p->ev_join) cudaEventDestroy(p->ev_join);
  if (p->ev_free) cudaEventDestroy(p->ev_free);
  for (cudaEvent_t e : p->ev_free_a)
    if (e) cudaEventDestroy(e);
  if (p->aux) cudaStreamDestroy(p->aux);
  if (p->have_phi) cufftDestroy(p->fft_phi);
  if (p->have_theta) cufftDestroy(p->fft_theta);
  if (!p->delta_shared) delta_free(p->delta);
  lane_tables_free(p->lane);
  void* ptrs[] = {p->U, p->Uf, p->W1, p->W2, p->W3, p->ph64, p->stage_in, p->stage_out, p->rc, p->rg};
  for (void* q : ptrs)
    if (q) cudaFree(q);
  delete p;
}

int create(ssht_plan_t* out, const ssht_plan_desc* desc, const DeltaWork* shared = nullptr) {
  if (!out || !desc) return fail(SSHT_EINVAL, "null argument");
  *out = nullptr;
  const int L = desc->L, s = desc->s, nfields = desc->batch;
  if (L < 1 || L > 2048) return fail(SSHT_EINVAL, "band-limit L must be in [1, 2048]");
  if (s <= -L || s >= L) return fail(SSHT_EINVAL, "spin must satisfy |s| < L");
  if (nfields < 1 || nfields > 65535) return fail(SSHT_EINVAL, "batch must be in [1, 65535]");
  if ((desc->flags & ~(SSHT_FLAG_REAL | SSHT_FLAG_RISBO | SSHT_FLAG_TUNE | SSHT_FLAG_SPIN_PAIR)) != 0)
    return fail(SSHT_EINVAL, "unknown flags");
  const bool pair = (desc->flags & SSHT_FLAG_SPIN_PAIR) != 0;
  if (pair && (desc->flags & SSHT_FLAG_REAL)) return fail(SSHT_EINVAL, "SSHT_FLAG_SPIN_PAIR and SSHT_FLAG_REAL exclude each other");
  if (pair && shared) return fail(SSHT_EINVAL, "groups take single fields, not spin pairs");
  const bool real = (desc->flags & SSHT_FLAG_REAL) != 0;
  if (real && s != 0) return fail(SSHT_EINVAL, "real fields (SSHT_FLAG_REAL) need spin 0");
  if (real && shared) return fail(SSHT_EINVAL, "groups take complex fields only");
  const int B = real ? (nfields + 1) / 2 : nfields;  // complex fields the transforms see
  if (desc->delta_mode != SSHT_DELTA_RECOMPUTE && desc->delta_mode != SSHT_DELTA_CACHE)
    return fail(SSHT_EINVAL, "unknown Delta mode");
  if (desc->precision != SSHT_FP64 && desc->precision != SSHT_FP32 && desc->precision != SSHT_TF32X3 &&
      desc->precision != SSHT_BF16X6)
    return fail(SSHT_EINVAL, "unknown precision");

  ssht_plan_t p = new (std::nothrow) ssht_plan_s();
  if (!p) return fail(SSHT_ENOMEM, "host allocation of the plan");
  int rc = 0;
  cudaError_t ce = cudaGetDevice(&p->device);
  if (ce == cudaSuccess) ce = cudaStreamCreateWithFlags(&p->aux, cudaStreamNonBlocking);
  if (ce == cudaSuccess) ce = cudaEventCreateWithFlags(&p->ev_fork, cudaEventDisableTiming);
  if (ce == cudaSuccess) ce = cudaEventCreateWithFlags(&p->ev_join, cudaEventDisableTiming);
  if (ce == cudaSuccess) ce = cudaEventCreateWithFlags(&p->ev_free, cudaEventDisableTiming);
  if (ce == cudaSuccess) ce = cudaEventCreateWithFlags(&p->ev_free_a[0], cudaEventDisableTiming);
  if (ce == cudaSuccess) ce = cudaEventCreateWithFlags(&p->ev_free_a[1], cudaEventDisableTiming);
  if (ce != cudaSuccess) {
    release(p);
    return fail(SSHT_ECUDA, std::string("plan stream/event setup: ") + cudaGetErrorString(ce));
  }
  p->d.L = L;
  p->d.Lp = L - 1;
  p->d.N = 2 * L - 1;
  p->s = s;
  p->B = B;
  p->precision = desc->precision;
  p->delta_mode = desc->delta_mode;
  p->real = real;
  p->nreal = real ? nfields : 0;
  p->pair = pair;
  p->f64 = desc->precision == SSHT_FP64;
  p->elem = p->f64 ? 16 : 8;
  const Dims& d = p->d;

  auto bail = [&](int code) {
    release(p);
    return code;
  };
  if (shared) {
    p->delta = *shared;
    p->delta_shared = true;
  } else {
    ce = delta_setup(p->delta, L, p->device, (desc->flags & SSHT_FLAG_RISBO) ? kDeltaRisbo : kDeltaColumn);
    if (ce != cudaSuccess) {
      release(p);
      return fail(ce == cudaErrorMemoryAllocation ? SSHT_ENOMEM : SSHT_ECUDA,
                  std::string("Delta recursion setup: ") + cudaGetErrorString(ce));
    }
    p->bytes += p->delta.bytes;
  }
  if (real && (ce = real_setup()) != cudaSuccess) {
    release(p);
    return fail(SSHT_ECUDA, std::string("real-field kernel attributes: ") + cudaGetErrorString(ce));
  }
  if ((rc = dalloc(p, (void**)&p->U, tri(L) * sizeof(double), "spin column"))) return bail(rc);
  if ((rc = dalloc(p, (void**)&p->Uf, tri(L) * sizeof(float), "spin column (FP32)"))) return bail(rc);
  // FP64: full N x N torus rows (the triangular forward's; the products' half rows, and L x L twice over, fit
  // but for L = 1) and the digits of a pass's data; FP32: half rows of N x L and the passes' operands (small
  // band-limits have none); tuning writes a contraction's output to the second workspace.
  const bool small = small_wanted(L, B, p->f64);
  const bool tensor = desc->precision == SSHT_TF32X3 || desc->precision == SSHT_BF16X6;
  TorusWork work;
  if (p->f64) {
    work.w1 = work.w2 = (size_t)B * std::max(d.N * d.N, 2) * p->elem;
  } else if (small) {
    work.w1 = (size_t)B * d.N * L * p->elem;
  } else {
    work = torus_work(L, B);
    p->torus_fields = work.fields;
  }
  if (tensor) work.w2 = std::max(work.w2, p->pair_coeff_bytes());
  if (pair && (rc = dalloc(p, &p->rc, (size_t)B * L * L * p->elem, "spin-pair coefficients"))) return bail(rc);
  if ((real || pair) && (ce = real_setup()) != cudaSuccess) {
    release(p);
    return fail(SSHT_ECUDA, std::string("packing kernel attributes: ") + cudaGetErrorString(ce));
  }
  if (real) {
    if ((rc = dalloc(p, &p->rc, p->pair_coeff_bytes(), "real-field pair coefficients"))) return bail(rc);
    if ((rc = dalloc(p, &p->rg, p->pair_grid_bytes(), "real-field pair samples"))) return bail(rc);
  }
  if ((rc = dalloc(p, &p->W1, work.w1, "torus workspace 1"))) return bail(rc);
  if ((rc = dalloc(p, &p->W2, work.w2, "torus workspace 2"))) return bail(rc);
  p->w_bytes = work.w1;
  const bool direct = p->f64 && !small && direct_wanted(L, B);
  p->contract_digits = p->f64 && !direct && !small && contract_digits_wanted(L, B);
  if (p->f64 && !direct && !small) {
    size_t w3 = digits_workspace_bytes(L, s, B);
    if (p->contract_digits) {
      w3 = std::max(w3, contract_digits_bytes(L, B));
      ce = cudaDeviceGetAttribute(&p->sms, cudaDevAttrMultiProcessorCount, p->device);
      if (ce == cudaSuccess) ce = contract_digits_setup();
      if (ce != cudaSuccess) {
        release(p);
        return fail(SSHT_ECUDA, std::string("contraction setup: ") + cudaGetErrorString(ce));
      }
    }
    if ((rc = dalloc(p, &p->W3, w3, "operand digits"))) return bail(rc);
    p->w3_bytes = w3;
  }
  if (p->f64) {
    // Phase table e^{i pi k / N}, |k| < N, computed in FP64 on the host.
    if ((rc = dalloc(p, (void**)&p->ph64, (size_t)(2 * d.N - 1) * sizeof(double2), "phase table"))) return bail(rc);
    std::vector<double2> h(2 * d.N - 1);
    const double pi = 3.14159265358979323846;
    for (int k = -(d.N - 1); k <= d.N - 1; ++k) {
      // reduce the angle to [-pi/2, pi/2]-ish before cos/sin for accuracy: k/N in (-1, 1)
      const double a = pi * (double)k / (double)d.N;
      h[k + d.N - 1] = make_double2(std::cos(a), std::sin(a));
    }
    ce = cudaMemcpy(p->ph64, h.data(), h.size() * sizeof(double2), cudaMemcpyHostToDevice);
    if (ce != cudaSuccess) {
      release(p);
      return fail(SSHT_ECUDA, std::string("phase table upload: ") + cudaGetErrorString(ce));
    }
    if ((rc = make_fft(p, &p->fft_phi, &p->have_phi, d.N, (size_t)B * d.L, "cuFFT phi plan"))) return bail(rc);
    if ((rc = make_fft(p, &p->fft_theta, &p->have_theta, d.N, (size_t)B * d.N, "cuFFT theta plan"))) return bail(rc);
  }
  ce = small    ? small_setup(&p->small, L, p->f64, p->device)
       : direct ? direct_setup(&p->direct, L)
       : p->f64 ? digits_setup(&p->digits, L, p->device)
                : torus_setup(&p->torus, L, p->device);
  if (ce != cudaSuccess) {
    release(p);
    return fail(ce == cudaErrorMemoryAllocation ? SSHT_ENOMEM : SSHT_ECUDA,
                std::string("torus pass setup: ") + cudaGetErrorString(ce));
  }
  p->bytes += small_bytes(p->small) + direct_bytes(p->direct) + digits_bytes(p->digits) + torus_bytes(p->torus);
  if (tensor) {
    ce = tc_setup(&p->tc, L, s, B, desc->precision == SSHT_BF16X6 ? 1 : 0, p->device);
    if (ce != cudaSuccess) {
      release(p);
      return fail(ce == cudaErrorMemoryAllocation ? SSHT_ENOMEM : SSHT_ECUDA,
                  std::string("tensor-core plan: ") + cudaGetErrorString(ce));
    }
    p->bytes += tc_bytes(p->tc);
  }
  if (tiles_direct(p)) {
    // the spin column once, from the table: a kept table, which ssht_wigner_delta hands out, is made whole (a group's
    // shared one is), and one of a small band-limit, whose sweep takes less than the list of tasks; else only the
    // entries that U reads (the sweep, L = 1024, s = 2: 0.95 -> 0.23 ms)
    if (p->delta_mode == SSHT_DELTA_CACHE || p->delta_shared || L <= 512) {
      if ((rc = run_delta(p, 0))) return bail(rc);
    } else {
      ce = column_run_spin(p->delta, L, s, 0);
      if (ce == cudaSuccess) ce = delta_spin_column(p->delta.table, L, s, p->U, p->Uf, 0);
      if (ce != cudaSuccess) {
        release(p);
        return fail(ce == cudaErrorMemoryAllocation ? SSHT_ENOMEM : SSHT_ECUDA, std::string("spin column: ") + cudaGetErrorString(ce));
      }
      p->launches += 2;
    }
    p->u_fixed = true;
    // the calls' recursions run on the plan's non-blocking stream: U must be complete first
    ce = cudaDeviceSynchronize();
    if (ce == cudaSuccess)
      ce = lane_tables_setup(p->lane, p->delta, L, s, p->Uf, tc_inverse_tiles(p->tc).nC, tc_a_tiles(p->tc).abase,
                             p->precision == SSHT_BF16X6);
    if (ce != cudaSuccess) {
      release(p);
      return fail(ce == cudaErrorMemoryAllocation ? SSHT_ENOMEM : SSHT_ECUDA,
                  std::string("spin column and recursion tables: ") + cudaGetErrorString(ce));
    }
    p->bytes += p->lane.bytes;
  }
  if (p->delta_mode == SSHT_DELTA_CACHE) {
    if (tiles_direct(p)) {
      if ((rc = make_operands(p, 0, 0)) || (rc = make_operands(p, 1, 0))) return bail(rc);
    } else {
      if ((rc = run_delta(p, 0))) return bail(rc);
      if (p->tc && ((rc = pack_a(p, 0, 0)) || (rc = pack_a(p, 1, 0)))) return bail(rc);
    }
    ce = cudaDeviceSynchronize();
    if (ce != cudaSuccess) {
      release(p);
      return fail(SSHT_ECUDA, std::string("Delta recursion: ") + cudaGetErrorString(ce));
    }
    int st = 0;
    cudaMemcpy(&st, p->delta.status, sizeof(int), cudaMemcpyDeviceToHost);
    if (st != 0) {
      release(p);
      return fail(SSHT_ETIMEOUT, "Delta recursion grid barrier timed out");
    }
    p->delta_ready = true;
  }
  if ((desc->flags & SSHT_FLAG_TUNE) && (rc = tune_tiles(p))) return bail(rc);
  *out = p;
  g_last_error.clear();
  return SSHT_OK;
}

}  // namespace

extern "C" {

int ssht_plan(ssht_plan_t* out, int L, int s, int batch) {
  ssht_plan_desc d{L, s, batch, SSHT_FP64, SSHT_DELTA_RECOMPUTE, 0};
  return create(out, &d);
}

int ssht_plan_ex(ssht_plan_t* out, const ssht_plan_desc* desc) { return create(out, desc); }

int ssht_plan_destroy(ssht_plan_t plan) {
  release(plan);
  return SSHT_OK;
}

int ssht_plan_workspace_bytes(ssht_plan_t plan, size_t* bytes) {
  if (!plan || !bytes) return fail(SSHT_EINVAL, "null argument");
  *bytes = plan->bytes;
  return SSHT_OK;
}

int ssht_inverse(ssht_plan_t p, const void* flm, void* f, void* stream) {
  if (!p) return fail(SSHT_EINVAL, "null plan");
  int rc = check_device(p);
  if (rc) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  if ((rc = set_streams(p, st))) return rc;
  IO io;
  // spin pairs from host memory: the inverse reads the coefficients of spin s only, so those alone cross the host
  // link, to where pair_gather would put them (L = 512, 24 pairs: 50 of 100 MB; inverse and forward 1.88 -> 1.63 ms)
  const bool half = p->pair && flm && f && !is_device_pointer(flm);
  if ((rc = io_begin(p, half ? p->rc : flm, p->coeff_bytes(), f, p->grid_bytes(), st, &io))) return rc;
  if (half) {
    const size_t n = (size_t)p->d.L * p->d.L * p->elem;
    SSHT_CUDA(cudaMemcpy2DAsync(p->rc, n, flm, 2 * n, n, p->B, cudaMemcpyHostToDevice, st), "input copy to device");
    rc = p->f64 ? inverse_impl<double>(p, p->rc, io.out_dev, st) : inverse_impl<float>(p, p->rc, io.out_dev, st);
  } else if (p->real)
    rc = p->f64 ? real_call<double>(p, 0, io.in_dev, io.out_dev, st) : real_call<float>(p, 0, io.in_dev, io.out_dev, st);
  else if (p->pair)
    rc = p->f64 ? pair_call<double>(p, 0, io.in_dev, io.out_dev, st) : pair_call<float>(p, 0, io.in_dev, io.out_dev, st);
  else
    rc = p->f64 ? inverse_impl<double>(p, io.in_dev, io.out_dev, st) : inverse_impl<float>(p, io.in_dev, io.out_dev, st);
  if (rc) return rc;
  return io_end(p, io, st);
}

int ssht_forward(ssht_plan_t p, const void* f, void* flm, void* stream) {
  if (!p) return fail(SSHT_EINVAL, "null plan");
  int rc = check_device(p);
  if (rc) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  if ((rc = set_streams(p, st))) return rc;
  IO io;
  if ((rc = io_begin(p, f, p->grid_bytes(), flm, p->coeff_bytes(), st, &io))) return rc;
  if (p->real)
    rc = p->f64 ? real_call<double>(p, 1, io.in_dev, io.out_dev, st) : real_call<float>(p, 1, io.in_dev, io.out_dev, st);
  else if (p->pair)
    rc = p->f64 ? pair_call<double>(p, 1, io.in_dev, io.out_dev, st) : pair_call<float>(p, 1, io.in_dev, io.out_dev, st);
  else
    rc = p->f64 ? forward_impl<double>(p, io.in_dev, io.out_dev, st) : forward_impl<float>(p, io.in_dev, io.out_dev, st);
  if (rc) return rc;
  return io_end(p, io, st);
}

int ssht_adjoint(ssht_plan_t p, const void* g, void* flm, void* stream) {
  if (!p) return fail(SSHT_EINVAL, "null plan");
  int rc = check_device(p);
  if (rc) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  if ((rc = set_streams(p, st))) return rc;
  IO io;
  if ((rc = io_begin(p, g, p->grid_bytes(), flm, p->coeff_bytes(), st, &io))) return rc;
  if (p->real)
    rc = p->f64 ? real_call<double>(p, 2, io.in_dev, io.out_dev, st) : real_call<float>(p, 2, io.in_dev, io.out_dev, st);
  else if (p->pair)
    rc = p->f64 ? pair_call<double>(p, 2, io.in_dev, io.out_dev, st) : pair_call<float>(p, 2, io.in_dev, io.out_dev, st);
  else
    rc = p->f64 ? adjoint_impl<double>(p, io.in_dev, io.out_dev, st) : adjoint_impl<float>(p, io.in_dev, io.out_dev, st);
  if (rc) return rc;
  return io_end(p, io, st);
}

int ssht_forward_triangular(ssht_plan_t p, const void* f, void* flm, void* stream) {
  if (!p) return fail(SSHT_EINVAL, "null plan");
  if (!p->f64) return fail(SSHT_EUNSUPPORTED, "the triangular forward is built for FP64 plans only");
  if (p->d.L > 2048) return fail(SSHT_EUNSUPPORTED, "band-limit too large for the triangular solve");
  int rc = check_device(p);
  if (rc) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  if ((rc = set_streams(p, st))) return rc;
  IO io;
  if ((rc = io_begin(p, f, p->grid_bytes(), flm, p->coeff_bytes(), st, &io))) return rc;
  const void* src = io.in_dev;
  void* dst = io.out_dev;
  if (p->real) {
    StageScope sc(p, SSHT_STAGE_PACK, st);
    SSHT_CUDA(real_pack_grid<double>(p->d.L, p->nreal, io.in_dev, p->rg, st), "real-field packing");
    p->launches += 1;
    src = p->rg;
    dst = p->rc;
  }
  if ((rc = begin_operands(p, 1, st))) return rc;
  if ((rc = analysis_front(p, src, st))) return rc;
  if ((rc = join_operands(p, st))) return rc;
  {
    StageScope sc(p, SSHT_STAGE_PROJECT, st);
    SSHT_CUDA(triangular_solve(p->d, p->s, p->B, p->delta.table, p->U, p->W1, p->ph64, dst, st), "triangular solve");
    p->launches += 2;
  }
  if ((rc = mark_free(p, st))) return rc;
  if (p->real) {
    StageScope sc(p, SSHT_STAGE_PACK, st);
    SSHT_CUDA(real_unpack_coeffs<double>(p->d.L, p->nreal, p->rc, io.out_dev, st), "real-field unpacking");
    p->launches += 1;
  }
  return io_end(p, io, st);
}

int ssht_wigner_delta(ssht_plan_t p, double* out, void* stream) {
  if (!p || !out) return fail(SSHT_EINVAL, "null argument");
  int rc = check_device(p);
  if (rc) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  if ((rc = ensure_delta(p, st))) return rc;
  const size_t bytes = delta_offset(p->d.L) * sizeof(double);
  if (is_device_pointer(out)) {
    SSHT_CUDA(cudaMemcpyAsync(out, p->delta.table, bytes, cudaMemcpyDeviceToDevice, st), "Delta table copy");
  } else {
    SSHT_CUDA(cudaMemcpyAsync(out, p->delta.table, bytes, cudaMemcpyDeviceToHost, st), "Delta table copy");
    SSHT_CUDA(cudaStreamSynchronize(st), "stream synchronize");
  }
  if ((rc = mark_free(p, st))) return rc;  // the recursion above ran on st: later calls wait for it
  SSHT_CUDA(cudaGetLastError(), "kernel launch");
  return SSHT_OK;
}

int ssht_plan_check(ssht_plan_t p) {
  if (!p) return fail(SSHT_EINVAL, "null plan");
  int rc = check_device(p);
  if (rc) return rc;
  SSHT_CUDA(cudaDeviceSynchronize(), "device synchronize");
  int st = 0;
  SSHT_CUDA(cudaMemcpy(&st, p->delta.status, sizeof(int), cudaMemcpyDeviceToHost), "status read");
  if (st != 0) {
    cudaMemset(p->delta.status, 0, sizeof(int));
    if (p->delta_mode == SSHT_DELTA_CACHE) p->delta_ready = false;
    return fail(SSHT_ETIMEOUT, std::string("a device-side wait exceeded its spin limit (") +
                                   ((st & kStatusBarrierTimeout) ? "recursion hand-off" : "") +
                                   ((st & kStatusBarrierTimeout) && (st & 2) ? ", " : "") +
                                   ((st & 2) ? "tensor-core pipeline" : "") + ")");
  }
  return SSHT_OK;
}

int ssht_plan_tile_config(ssht_plan_t p, int* cfg) {
  if (!p || !cfg) return fail(SSHT_EINVAL, "null argument");
  if (!p->tc) return fail(SSHT_EUNSUPPORTED, "the plan has no tensor-core contraction");
  const TcConfig c = tc_config(p->tc);
  cfg[0] = c.slice;
  cfg[1] = c.stages;
  cfg[2] = c.inv_order;
  cfg[3] = c.fwd_order;
  return SSHT_OK;
}

int ssht_plan_set_wait_limit(ssht_plan_t p, long long ns) {
  if (!p) return fail(SSHT_EINVAL, "null plan");
  p->wait_ns = ns > 0 ? ns : kDefaultWaitNs;
  return SSHT_OK;
}

int ssht_plan_profile(ssht_plan_t p, int enable) {
  if (!p) return fail(SSHT_EINVAL, "null plan");
  int rc = check_device(p);
  if (rc) return rc;
  SSHT_CUDA(cudaDeviceSynchronize(), "device synchronize");
  for (auto& e : p->evs) {
    cudaEventDestroy(e.a);
    cudaEventDestroy(e.b);
  }
  p->evs.clear();
  for (int i = 0; i < SSHT_NUM_STAGES; ++i) {
    p->prof_ms[i] = 0.0;
    p->prof_n[i] = 0;
  }
  p->prof = enable != 0;
  return SSHT_OK;
}

int ssht_plan_profile_read(ssht_plan_t p, double* ms, long long* count, int nstages, long long* launches) {
  if (!p) return fail(SSHT_EINVAL, "null plan");
  if (nstages < 0 || nstages > SSHT_NUM_STAGES || (nstages > 0 && (!ms || !count)))
    return fail(SSHT_EINVAL, "bad stage buffers");
  int rc = check_device(p);
  if (rc) return rc;
  SSHT_CUDA(cudaDeviceSynchronize(), "device synchronize");
  fold_events(p);
  for (int i = 0; i < nstages; ++i) {
    ms[i] = p->prof_ms[i];
    count[i] = p->prof_n[i];
  }
  if (launches) *launches = p->launches;
  return SSHT_OK;
}

int ssht_plan_profile_trace(ssht_plan_t p, int* stage, int* lane, double* t0, double* t1, int cap, int* n) {
  if (!p) return fail(SSHT_EINVAL, "null plan");
  if (!n || cap < 0 || (cap > 0 && (!stage || !lane || !t0 || !t1))) return fail(SSHT_EINVAL, "bad trace buffers");
  int rc = check_device(p);
  if (rc) return rc;
  SSHT_CUDA(cudaDeviceSynchronize(), "device synchronize");
  *n = (int)std::min(p->evs.size(), (size_t)cap);
  double first = 0.0;  // brackets of the two streams need not start in recording order
  for (int i = 0; i < *n; ++i) {
    const auto& e = p->evs[i];
    float a = 0.f, b = 0.f;
    SSHT_CUDA(cudaEventElapsedTime(&a, p->evs[0].a, e.a), "trace event time");
    SSHT_CUDA(cudaEventElapsedTime(&b, p->evs[0].a, e.b), "trace event time");
    stage[i] = e.stage;
    lane[i] = e.lane;
    t0[i] = a;
    t1[i] = b;
    first = std::min(first, (double)a);
  }
  for (int i = 0; i < *n; ++i) {
    t0[i] -= first;
    t1[i] -= first;
  }
  fold_events(p);
  return SSHT_OK;
}

const char* ssht_last_error(void) { return g_last_error.c_str(); }

int ssht_debug_fail_allocation(int n) {
  if (n < 0) return fail(SSHT_EINVAL, "ssht_debug_fail_allocation: n must be >= 0");
  g_alloc_countdown.store(n);
  return SSHT_OK;
}

int ssht_debug_bounds(long long* count, int* site, long long* index, long long* extent) {
  if (!kBoundsChecked) return fail(SSHT_EUNSUPPORTED, "ssht_debug_bounds: this library was built without index checks");
  SSHT_CUDA(cudaDeviceSynchronize(), "synchronize");
  cudaError_t (*take[])(BoundsRecord*) = {bounds_take_torus_pass,   bounds_take_torus_small,     bounds_take_torus_direct,
                                          bounds_take_torus_digits, bounds_take_contract_digits, bounds_take_contract_tc,
                                          bounds_take_delta_column, bounds_take_real,            bounds_take_contract_simt};
  BoundsRecord first{};
  long long total = 0;
  for (auto f : take) {
    BoundsRecord r{};
    SSHT_CUDA(f(&r), "index-check record");
    if (r.count && !total) first = r;
    total += (long long)r.count;
  }
  if (count) *count = total;
  if (site) *site = total ? first.kernel : 0;
  if (index) *index = total ? first.index : 0;
  if (extent) *extent = total ? first.extent : 0;
  return 0;
}

int ssht_version(void) { return 100; }

}  // extern "C"

// ---------------------------------------------------------------------------------------------
// Groups: many fields of uneven band-limit and spin in one call (and one CUDA graph).
//
// Fields are bucketed by (L, s); each bucket is one plan over its fields, which sit contiguously
// in the caller's flat buffers in group order (ssht_group_layout).  CUDA-core buckets
// of one L share one Delta table: in recompute mode each call runs one recursion per such L, on its
// own stream, and the buckets wait for it before their spin column; in cache mode the tables are
// made once here.  Tensor-core buckets write their own tiles (tiles_direct): with 256 fields of L in
// {128, .., 1024} and 20 buckets, packing every bucket's tiles from shared tables made a step
// (inverse and forward) 39.1 ms, the sweeps into the tiles 29.4.  Buckets run on their own streams, forked from and joined to the caller's.
// With tuning on, each bucket times every contraction form of the group's precision class
// (FP32, split-FP16, split-BF16 for FP32-class groups; the tensor-core forms with their own tuned
// shape) on its own shape and keeps the fastest.
// ---------------------------------------------------------------------------------------------

struct ssht_group_s {
  int device = 0;
  int n = 0;
  int precision = 0, delta_mode = 0;
  size_t elem = 8;
  std::vector<int> order;            // group position -> caller's field index
  std::vector<long long> coff, goff; // per group position: element offsets of coefficients / samples
  struct Holder {
    int L = 0;
    DeltaWork dw{};
    cudaEvent_t ev = nullptr;
    bool table_used = false;  // some bucket of this L contracts from the table (CUDA-core plans)
  };
  // The shared recursions run one after another on one stream: each is a cooperative grid over
  // every SM, so running two at once would only make them wait for each other's SMs.
  cudaStream_t rec_st = nullptr;
  std::vector<Holder> holders;
  struct Bucket {
    int L = 0, s = 0, first = 0, count = 0, holder = 0;
    ssht_plan_t plan = nullptr;
    cudaStream_t st = nullptr;
    cudaEvent_t ev = nullptr;
  };
  std::vector<Bucket> buckets;
  cudaEvent_t ev_start = nullptr;
  cudaGraphExec_t exec = nullptr;
};

namespace {

void group_release(ssht_group_t g) {
  if (!g) return;
  cudaDeviceSynchronize();
  if (g->exec) cudaGraphExecDestroy(g->exec);
  for (auto& b : g->buckets) {
    if (b.plan) release(b.plan);
    if (b.st) cudaStreamDestroy(b.st);
    if (b.ev) cudaEventDestroy(b.ev);
  }
  for (auto& h : g->holders) {
    delta_free(h.dw);
    if (h.ev) cudaEventDestroy(h.ev);
  }
  if (g->rec_st) cudaStreamDestroy(g->rec_st);
  if (g->ev_start) cudaEventDestroy(g->ev_start);
  delete g;
}

// One call of every bucket; which: 0 inverse, 1 forward, 2 adjoint.
int group_call(ssht_group_t g, int which, const void* in, void* out, cudaStream_t st) {
  SSHT_CUDA(cudaEventRecord(g->ev_start, st), "group fork");
  if (g->delta_mode == SSHT_DELTA_RECOMPUTE) {
    // recursions into a shared table only for the band-limits whose buckets read it (a forked
    // stream that nothing joins would spoil a capture)
    bool forked = false;
    for (auto& h : g->holders) {
      if (!h.table_used) continue;
      if (!forked) SSHT_CUDA(cudaStreamWaitEvent(g->rec_st, g->ev_start, 0), "group fork wait");
      forked = true;
      SSHT_CUDA(delta_run(h.dw, h.L, g->rec_st), "shared Delta recursion");
      SSHT_CUDA(cudaEventRecord(h.ev, g->rec_st), "shared Delta event");
    }
  }
  for (auto& b : g->buckets) {
    ssht_plan_t p = b.plan;
    SSHT_CUDA(cudaStreamWaitEvent(b.st, g->ev_start, 0), "group fork wait");
    p->delta_event = g->delta_mode == SSHT_DELTA_RECOMPUTE && g->holders[b.holder].table_used ? g->holders[b.holder].ev : nullptr;
    int rc = set_streams(p, b.st);
    if (rc) return rc;
    const long long ci = g->coff[b.first], gi = g->goff[b.first];
    const char* src = (const char*)in + (which == 0 ? ci : gi) * g->elem;
    char* dst = (char*)out + (which == 0 ? gi : ci) * g->elem;
    if (which == 0)
      rc = p->f64 ? inverse_impl<double>(p, src, dst, b.st) : inverse_impl<float>(p, src, dst, b.st);
    else if (which == 1)
      rc = p->f64 ? forward_impl<double>(p, src, dst, b.st) : forward_impl<float>(p, src, dst, b.st);
    else
      rc = p->f64 ? adjoint_impl<double>(p, src, dst, b.st) : adjoint_impl<float>(p, src, dst, b.st);
    if (rc) return rc;
    SSHT_CUDA(cudaEventRecord(b.ev, b.st), "group join event");
  }
  for (auto& b : g->buckets) SSHT_CUDA(cudaStreamWaitEvent(st, b.ev, 0), "group join wait");
  return 0;
}

// Mean milliseconds of inverse + forward of one plan on zero data (shapes decide the time).
int time_plan(ssht_plan_t p, float* ms) {
  void *a = nullptr, *b = nullptr, *c = nullptr;
  const size_t cb = p->coeff_bytes(), gb = p->grid_bytes();
  int rc = 0;
  if ((rc = dalloc(p, &a, cb, "tuning input")) || (rc = dalloc(p, &b, gb, "tuning grid")) ||
      (rc = dalloc(p, &c, cb, "tuning output"))) {
    cudaFree(a);
    cudaFree(b);
    return rc;
  }
  p->bytes -= cb + gb + cb;
  cudaEvent_t e0, e1;
  cudaStream_t st = nullptr;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking);
  cudaMemsetAsync(a, 0, cb, st);
  for (int it = 0; it < 6 && !rc; ++it) {
    if (it == 2) cudaEventRecord(e0, st);
    rc = p->f64 ? inverse_impl<double>(p, a, b, st) : inverse_impl<float>(p, a, b, st);
    if (!rc) rc = p->f64 ? forward_impl<double>(p, b, c, st) : forward_impl<float>(p, b, c, st);
  }
  cudaEventRecord(e1, st);
  cudaEventSynchronize(e1);
  float t = 0.f;
  cudaEventElapsedTime(&t, e0, e1);
  *ms = t / 4.f;
  cudaStreamDestroy(st);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaFree(a);
  cudaFree(b);
  cudaFree(c);
  return rc;
}

int group_create(ssht_group_t* out, int n, const int* Ls, const int* ss, int precision, int delta_mode, int tune) {
  if (!out || !Ls || !ss) return fail(SSHT_EINVAL, "null argument");
  *out = nullptr;
  if (n < 1) return fail(SSHT_EINVAL, "a group needs at least one field");
  if (precision != SSHT_FP64 && precision != SSHT_FP32 && precision != SSHT_TF32X3 && precision != SSHT_BF16X6)
    return fail(SSHT_EINVAL, "unknown precision");
  if (delta_mode != SSHT_DELTA_RECOMPUTE && delta_mode != SSHT_DELTA_CACHE) return fail(SSHT_EINVAL, "unknown Delta mode");
  for (int i = 0; i < n; ++i) {
    if (Ls[i] < 1 || Ls[i] > 2048) return fail(SSHT_EINVAL, "band-limit L must be in [1, 2048]");
    if (ss[i] <= -Ls[i] || ss[i] >= Ls[i]) return fail(SSHT_EINVAL, "spin must satisfy |s| < L");
  }
  ssht_group_t g = new (std::nothrow) ssht_group_s();
  if (!g) return fail(SSHT_ENOMEM, "host allocation of the group");
  auto bail = [&](int code) {
    group_release(g);
    return code;
  };
  cudaError_t ce = cudaGetDevice(&g->device);
  if (ce == cudaSuccess) ce = cudaEventCreateWithFlags(&g->ev_start, cudaEventDisableTiming);
  if (ce == cudaSuccess) ce = cudaStreamCreateWithFlags(&g->rec_st, cudaStreamNonBlocking);
  if (ce != cudaSuccess) return bail(fail(SSHT_ECUDA, std::string("group setup: ") + cudaGetErrorString(ce)));
  g->n = n;
  g->precision = precision;
  g->delta_mode = delta_mode;
  g->elem = precision == SSHT_FP64 ? 16 : 8;
  // group order: by L, then s, then the caller's index
  g->order.resize(n);
  for (int i = 0; i < n; ++i) g->order[i] = i;
  std::stable_sort(g->order.begin(), g->order.end(),
                   [&](int a, int b) { return Ls[a] != Ls[b] ? Ls[a] < Ls[b] : ss[a] < ss[b]; });
  g->coff.resize(n + 1);
  g->goff.resize(n + 1);
  long long c = 0, q = 0;
  for (int k = 0; k < n; ++k) {
    const int L = Ls[g->order[k]];
    g->coff[k] = c;
    g->goff[k] = q;
    c += (long long)L * L;
    q += (long long)L * (2 * L - 1);
  }
  g->coff[n] = c;
  g->goff[n] = q;
  // shared Delta tables, one per distinct L
  for (int k = 0; k < n; ++k) {
    const int L = Ls[g->order[k]];
    if (g->holders.empty() || g->holders.back().L != L) {
      g->holders.emplace_back();
      auto& h = g->holders.back();
      h.L = L;
      ce = delta_setup(h.dw, L, g->device);
      if (ce == cudaSuccess) ce = cudaEventCreateWithFlags(&h.ev, cudaEventDisableTiming);
      if (ce == cudaSuccess) ce = delta_run(h.dw, L, 0);  // valid tables for tuning and cache mode
      if (ce != cudaSuccess)
        return bail(fail(ce == cudaErrorMemoryAllocation ? SSHT_ENOMEM : SSHT_ECUDA,
                         std::string("shared Delta setup: ") + cudaGetErrorString(ce)));
    }
  }
  ce = cudaDeviceSynchronize();
  if (ce != cudaSuccess) return bail(fail(SSHT_ECUDA, std::string("shared Delta: ") + cudaGetErrorString(ce)));
  // buckets
  for (int k = 0; k < n;) {
    const int L = Ls[g->order[k]], s = ss[g->order[k]];
    int e = k;
    while (e < n && Ls[g->order[e]] == L && ss[g->order[e]] == s) ++e;
    g->buckets.emplace_back();
    auto& b = g->buckets.back();
    b.L = L;
    b.s = s;
    b.first = k;
    b.count = e - k;
    b.holder = (int)g->holders.size() - 1;
    while (g->holders[b.holder].L != L) --b.holder;
    ce = cudaStreamCreateWithFlags(&b.st, cudaStreamNonBlocking);
    if (ce == cudaSuccess) ce = cudaEventCreateWithFlags(&b.ev, cudaEventDisableTiming);
    if (ce != cudaSuccess) return bail(fail(SSHT_ECUDA, "bucket stream setup"));
    std::vector<int> cands;
    if (!tune || precision == SSHT_FP64) {
      cands.push_back(precision);
    } else {
      cands.push_back(SSHT_FP32);
      cands.push_back(SSHT_TF32X3);
      cands.push_back(SSHT_BF16X6);
    }
    float best = 0.f;
    for (int cand : cands) {
      ssht_plan_desc d{L, s, b.count, cand, delta_mode,
                       (tune && (cand == SSHT_TF32X3 || cand == SSHT_BF16X6)) ? SSHT_FLAG_TUNE : 0};
      ssht_plan_t p = nullptr;
      int rc = create(&p, &d, &g->holders[b.holder].dw);
      if (rc) return bail(rc);
      float ms = 0.f;
      if (cands.size() > 1 && (rc = time_plan(p, &ms))) {
        release(p);
        return bail(rc);
      }
      if (!b.plan || ms < best) {
        if (b.plan) release(b.plan);
        b.plan = p;
        best = ms;
      } else {
        release(p);
      }
    }
    if (!tiles_direct(b.plan)) g->holders[b.holder].table_used = true;
    k = e;
  }
  *out = g;
  g_last_error.clear();
  return SSHT_OK;
}

}  // namespace

extern "C" {

int ssht_group_create(ssht_group_t* out, int n, const int* L, const int* s, int precision, int delta_mode, int tune) {
  return group_create(out, n, L, s, precision, delta_mode, tune);
}

int ssht_group_destroy(ssht_group_t g) {
  group_release(g);
  return SSHT_OK;
}

int ssht_group_layout(ssht_group_t g, int* order, long long* coeff_offset, long long* grid_offset) {
  if (!g) return fail(SSHT_EINVAL, "null group");
  for (int k = 0; k < g->n; ++k) {
    if (order) order[k] = g->order[k];
    if (coeff_offset) coeff_offset[k] = g->coff[k];
    if (grid_offset) grid_offset[k] = g->goff[k];
  }
  if (coeff_offset) coeff_offset[g->n] = g->coff[g->n];
  if (grid_offset) grid_offset[g->n] = g->goff[g->n];
  return SSHT_OK;
}

int ssht_group_buckets(ssht_group_t g, int* nbuckets, int* L, int* s, int* count, int* precision) {
  if (!g || !nbuckets) return fail(SSHT_EINVAL, "null argument");
  const int nb = (int)g->buckets.size();
  const int cap = *nbuckets;
  *nbuckets = nb;
  for (int i = 0; i < nb && i < cap; ++i) {
    if (L) L[i] = g->buckets[i].L;
    if (s) s[i] = g->buckets[i].s;
    if (count) count[i] = g->buckets[i].count;
    if (precision) precision[i] = g->buckets[i].plan->precision;
  }
  return SSHT_OK;
}

int ssht_group_bucket_tile_config(ssht_group_t g, int bucket, int* cfg) {
  if (!g || !cfg) return fail(SSHT_EINVAL, "null argument");
  if (bucket < 0 || bucket >= (int)g->buckets.size()) return fail(SSHT_EINVAL, "no such bucket");
  return ssht_plan_tile_config(g->buckets[bucket].plan, cfg);
}

static int group_entry(ssht_group_t g, int which, const void* in, void* out, void* stream) {
  if (!g || !in || !out) return fail(SSHT_EINVAL, "null argument");
  int cur = -1;
  SSHT_CUDA(cudaGetDevice(&cur), "cudaGetDevice");
  if (cur != g->device) return fail(SSHT_EINVAL, "group used on another device");
  if (!is_device_pointer(in) || !is_device_pointer(out)) return fail(SSHT_EINVAL, "group buffers must be device memory");
  return group_call(g, which, in, out, (cudaStream_t)stream);
}

int ssht_group_inverse(ssht_group_t g, const void* flm, void* f, void* stream) { return group_entry(g, 0, flm, f, stream); }
int ssht_group_forward(ssht_group_t g, const void* f, void* flm, void* stream) { return group_entry(g, 1, f, flm, stream); }
int ssht_group_adjoint(ssht_group_t g, const void* f, void* flm, void* stream) { return group_entry(g, 2, f, flm, stream); }

int ssht_group_capture(ssht_group_t g, const void* flm, void* f, void* flm_out, void* stream) {
  if (!g || !flm || !f || !flm_out) return fail(SSHT_EINVAL, "null argument");
  if (!is_device_pointer(flm) || !is_device_pointer(f) || !is_device_pointer(flm_out))
    return fail(SSHT_EINVAL, "group buffers must be device memory");
  (void)stream;  // capturing launches nothing: it records on a private stream (the legacy default
                 // stream cannot be captured)
  cudaStream_t cap = nullptr;
  SSHT_CUDA(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking), "capture stream");
  if (g->exec) {
    cudaGraphExecDestroy(g->exec);
    g->exec = nullptr;
  }
  cudaGraph_t graph = nullptr;
  cudaError_t ce = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
  int rc = 0;
  if (ce == cudaSuccess) {
    rc = group_call(g, 0, flm, f, cap);
    if (!rc) rc = group_call(g, 1, f, flm_out, cap);
    ce = cudaStreamEndCapture(cap, &graph);
  }
  if (ce == cudaSuccess && !rc) ce = cudaGraphInstantiate(&g->exec, graph, 0);
  if (graph) cudaGraphDestroy(graph);
  cudaStreamDestroy(cap);
  if (rc) return rc;
  if (ce != cudaSuccess) return fail(SSHT_ECUDA, std::string("group graph capture: ") + cudaGetErrorString(ce));
  return SSHT_OK;
}

int ssht_group_replay(ssht_group_t g, void* stream) {
  if (!g || !g->exec) return fail(SSHT_EINVAL, "no captured graph");
  SSHT_CUDA(cudaGraphLaunch(g->exec, (cudaStream_t)stream), "graph launch");
  return SSHT_OK;
}

int ssht_group_check(ssht_group_t g) {
  if (!g) return fail(SSHT_EINVAL, "null group");
  SSHT_CUDA(cudaDeviceSynchronize(), "device synchronize");
  for (auto& h : g->holders) {
    int st = 0;
    SSHT_CUDA(cudaMemcpy(&st, h.dw.status, sizeof(int), cudaMemcpyDeviceToHost), "status read");
    if (st != 0) {
      cudaMemset(h.dw.status, 0, sizeof(int));
      return fail(SSHT_ETIMEOUT, "a Delta recursion wait exceeded its spin limit");
    }
  }
  return SSHT_OK;
}

}  // extern "C"
