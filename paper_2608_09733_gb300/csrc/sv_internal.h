// sv_internal.h -- structures shared by the host planner (sv_plan.cpp, sv_api.cpp)
// and the CUDA kernels (sv_sweep.cu, sv_reduce.cu).  Not part of the public ABI.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <complex>
#include <initializer_list>
#include <memory>
#include <shared_mutex>
#include <string>
#include <vector>

#include "../../include/sv.h"
#include "sv_prog_layout.h"

namespace sv {

using cplx = std::complex<double>;

// ----------------------------------------------------------------- host plan

// The coefficients of one operation: a vector whose first four entries (a
// one-qubit matrix, a two-qubit diagonal) need no allocation.  A plan copies
// its operations a few times, and most of them are that small.
class Coefs {
 public:
  Coefs() = default;
  Coefs(std::initializer_list<cplx> l) { assign(l.begin(), l.end()); }
  Coefs(size_t n, cplx v) { assign(n, v); }
  Coefs(const Coefs& o) { assign(o.begin(), o.end()); }
  Coefs(Coefs&& o) noexcept { take(o); }
  Coefs& operator=(const Coefs& o) {
    if (this != &o) assign(o.begin(), o.end());
    return *this;
  }
  Coefs& operator=(Coefs&& o) noexcept {
    if (this != &o) take(o);
    return *this;
  }
  // [b, e) must not point into this object
  void assign(const cplx* b, const cplx* e) { std::copy(b, e, room((size_t)(e - b))); }
  void assign(size_t n, cplx v) { std::fill_n(room(n), n, v); }
  void clear() { n_ = 0; }
  size_t size() const { return n_; }
  cplx* data() { return at_; }
  const cplx* data() const { return at_; }
  cplx* begin() { return at_; }
  cplx* end() { return at_ + n_; }
  const cplx* begin() const { return at_; }
  const cplx* end() const { return at_ + n_; }
  cplx& operator[](size_t i) { return at_[i]; }
  const cplx& operator[](size_t i) const { return at_[i]; }
  bool operator==(const Coefs& o) const { return n_ == o.n_ && std::equal(begin(), end(), o.begin()); }

 private:
  static constexpr size_t kSmall = 4;
  cplx* room(size_t n) {
    if (n > cap_) {
      big_.reset(new cplx[n]);
      at_ = big_.get();
      cap_ = n;
    }
    n_ = n;
    return at_;
  }
  void take(Coefs& o) {
    if (o.big_) {
      big_ = std::move(o.big_);
      at_ = big_.get();
      cap_ = o.cap_;
      n_ = o.n_;
      o.at_ = o.small_;
      o.cap_ = kSmall;
    } else {
      assign(o.begin(), o.end());
    }
    o.n_ = 0;
  }
  size_t n_ = 0, cap_ = kSmall;
  cplx* at_ = small_;
  cplx small_[kSmall];
  std::unique_ptr<cplx[]> big_;
};

// A gate after lowering (a matrix in double precision) or a fused block.
struct LOp {
  OpKind kind = OPK_DENSE;
  int8_t k = 0;                   // matrix qubits
  int8_t q[5] = {0, 0, 0, 0, 0};  // global matrix qubits, q[0] = least significant matrix bit
  int8_t nc = 0;
  int8_t c[5] = {0, 0, 0, 0, 0};   // global control qubits
  int8_t cs[5] = {1, 1, 1, 1, 1};  // required control states
  Coefs m;                   // DENSE/REAL: 2^k x 2^k row-major; DIAG: 2^k; ANTIDIAG: {a, b}
  uint64_t touch = 0;        // every qubit the op reads (matrix qubits and controls)
  uint64_t need = 0;         // qubits that must be inside the tile
  int first_gate = 0;        // index of the first source gate (fusion bookkeeping)
};

struct Sweep {
  int m = 0, L = 0;
  int tq[kMaxTileQ];
  std::vector<int> ops;      // indices into the LOp list, in application order
};

struct Plan {
  int n = 0;
  std::vector<LOp> ops;
  std::vector<int> block_starts;  // first gate of each op (fusion blocks) + n_gates
  std::vector<Sweep> sweeps;
  bool lane = false;        // passes of the cluster kernel (sv_lane.cu): tiles of up to 2^14 amplitudes
  // programs whose ops may be reordered over their phases and whose phase
  // tables are carried across bit flips and swaps (permuted) instead of applied
  // before them; not the packed and session programs, whose rounding stays as
  // it is
  bool carry_flips = false;
};

// Errors carry a status and a message up to the C ABI.
struct Error {
  sv_status status;
  std::string msg;
};

[[noreturn]] inline void fail(sv_status s, const std::string& m) { throw Error{s, m}; }
inline void cuda_check(cudaError_t e, const char* what) {
  if (e != cudaSuccess) fail(SV_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}
void set_last_error(const std::string& m);

// Runs f, mapping sv::Error and host exceptions to an sv_status.
template <typename F>
sv_status guarded(F&& f) {
  try {
    f();
    return SV_OK;
  } catch (const Error& e) {
    set_last_error(e.msg);
    return e.status;
  } catch (const std::bad_alloc&) {
    set_last_error("host allocation failed");
    return SV_ERR_OOM;
  } catch (...) {
    set_last_error("unexpected host exception");
    return SV_ERR_INVALID;
  }
}

// Device pointer checks (device/managed memory of the current device, 16-byte
// aligned, inside its allocation) and library-owned scratch: one grow-only
// buffer per (device, stream, name).
void check_device_buffer(const void* p, size_t bytes, const char* what);
void* scratch_buffer(cudaStream_t stream, const char* name, size_t bytes);

// Pinned host staging per (device, stream, name), grow-only; `ready` is
// recorded after the last copy out of it, so a rewrite waits for that copy.
struct Pinned {
  void* p = nullptr;
  size_t cap = 0;
  cudaEvent_t ready = nullptr;
};
Pinned& pinned_buffer(cudaStream_t stream, const char* name, size_t bytes);

// Lowering (gate records -> double-precision matrices), the paper's greedy
// fusion, and the tile scheduler.  Throw sv::Error on invalid input.
void validate_gates(int n, const sv_gate* gates, size_t n_gates, size_t n_param_values);
Coefs gate_matrix(const sv_gate& g, const double* param_values);
LOp lower_gate(const sv_gate& g, const double* param_values, int index);
std::vector<LOp> fuse_greedy(int n, const sv_gate* gates, size_t n_gates, const double* param_values, int kmax,
                             std::vector<int>* block_starts, bool dense_always);
void classify(LOp& op);
std::vector<Sweep> schedule_sweeps(int n, const std::vector<const LOp*>& ops, int tile_q, int low_q, int coef_pool,
                                   int ops_per_pass, bool commute);
Plan make_plan(int n, sv_dtype dtype, const sv_gate* gates, size_t n_gates, const double* param_values,
               size_t n_param_values, const sv_exec_opts& opts, int tile_q_override = 0, bool lane = false);
// Whether a state of this size with these options takes the cluster pass.
bool lane_sizes(int n, const sv_exec_opts& opts);
double op_cost(const LOp& op);
int tile_qubits_for(sv_dtype dtype, int n);
int low_qubits_for(sv_dtype dtype);
int reg_qubits_for(int m);  // register qubits of a tile of m qubits (4, or 5 for m >= 12)

// The kernel program of one sweep (sv_program.cpp); rq_override > 0 forces the
// register qubits of the register phases.
// A 2x2 unitary U written as g * diag(1, ephi) * [[C, -S], [S, C]] * diag(1, elam)
// (the Z-Y-Z Euler form, C = cos(alpha), S = sin(alpha), alpha in [0, pi/2]);
// false if the reconstruction misses U by more than tol in any entry.
struct RotSplit {
  cplx g = 1.0, ephi = 1.0, elam = 1.0;
  double C = 1.0, S = 0.0;
};
bool rot_split(const cplx* U, double tol, RotSplit& r);

// An op as the phases see it: the qubits it acts on other than diagonally and
// diagonally (controls, diagonals), the local positions it needs as register
// slots, and whether it runs in shared memory (a phase of its own).
struct PhaseOp {
  uint64_t moves, holds;
  uint32_t need;
  bool smem;
};
PhaseOp phase_op(const LOp& op, uint32_t need, bool smem);
// The ops of a pass ordered by phases of rq register slots: a phase takes, in
// order, every op whose slots still fit and that commutes with each op passed
// over before it.  *phases: the phases of that order; *runs: of the given
// order, a phase ending at the first op that does not fit.
std::vector<int> order_by_phase(const std::vector<PhaseOp>& ops, int rq, int* phases, int* runs);

// The device programs of a plan's passes, appended to `out`: one a pass, more
// where a pass does not fit one.
template <typename R>
void build_programs(const Plan& plan, std::vector<SweepProgram<R>>& out, int rq_override = 0);
// How many build_programs makes (the passes that run), building only those that
// could be more than one.
template <typename R>
size_t count_programs(const Plan& plan);

// ----------------------------------------------------------------- launches
// (sv_sweep.cu / sv_reduce.cu).  All return cudaError_t of the launch.

// *kernel (if not NULL) names the pass kernel that ran: "sweep_jit" (the
// program's own compiled kernel, TMA tile movement), "sweep_tma" (TMA, the
// interpreting kernel) or "sweep" (cp.async).  jit (if not NULL) is the
// program's compiled kernel, used wherever the TMA pass runs.
struct JitKernel;
template <typename R>
cudaError_t launch_sweep(Cx<R>* state, const SweepProgram<R>& prog, cudaStream_t stream,
                         const char** kernel = nullptr, const JitKernel* jit = nullptr);
// The cluster pass of small states (sv_lane.cu); whether the current device
// takes it now (clusters of 16 CTAs, which a live serving session's resident
// CTAs could keep waiting, so not beside one).
template <typename R>
cudaError_t launch_lane_pass(Cx<R>* state, const SweepProgram<R>& prog, cudaStream_t stream);
bool lane_pass_available();
template <typename R>
cudaError_t launch_init_basis(Cx<R>* state, int n, uint64_t index, cudaStream_t stream);
// One CTA per small request (whole state in shared memory): request b runs
// programs first_prog[b] .. first_prog[b+1]-1 (program p at buf + offset[p],
// device memory) and writes sum_q <Z_q> to out[b].
template <typename R>
cudaError_t launch_small_batch(const char* buf, const uint64_t* offset, const int* first_prog, const int* nq, int n_requests,
                               int max_n, double* out, cudaStream_t stream);

// Dynamic shared memory of a session's CTA, whose largest state has max_n
// qubits: that state.
constexpr size_t small_session_smem(size_t amp_bytes, int max_n) { return amp_bytes << max_n; }

// Persistent packed small states (serving sessions, sv_serve.cpp).  The
// entries, published count, exit flag, results and done words are pinned host
// memory mapped into the device; head and status are device memory.
struct SmallEntry {
  int32_t first_prog, last_prog;  // the request's programs in the session's program arena
  int32_t n_qubits, slot;         // state size; result slot (results[slot], done[slot])
};
struct SmallSessionDev {
  const SmallEntry* entries;      // ring of `capacity` entries; ticket t uses entries[t % capacity]
  const long long* tail;          // tickets published so far (written by the host)
  const int* exit_flag;           // nonzero: end the session once no published ticket is left
  unsigned long long* head;       // next ticket to claim (device)
  double* results;                // sum_q <Z_q> per slot
  long long* done;                // done[slot] = ticket + 1 once results[slot] is written
  int* status;                    // SV_OK, or SV_ERR_TIMEOUT when a wait ran out (device)
  long long capacity;
  uint64_t limit_ns;              // longest wait for a ticket
};
template <typename R>
cudaError_t launch_small_session(const SmallSessionDev& d, const SweepProgram<R>* progs, int max_n, int grid,
                                 cudaStream_t stream);
// Live sessions per device and their resident CTAs.  A session's CTAs hold
// their SMs, so while one is live the TMA pass (one CTA per SM, a fixed share
// of tiles each) launches on the SMs the sessions leave free.
void session_opened(int device, int ctas);
void session_closed(int device, int ctas);
bool session_live(int device);
// Held shared while a cluster pass is enqueued, exclusively while a session starts.
std::shared_mutex& session_gate();
// Ends the kernels of the device's live sessions and holds them (their locks)
// until sessions_release, which relaunches those with requests not done
// (sv_serve.cpp): a module load waits for every resident kernel to end.
void sessions_quiesce(int device, std::vector<sv_small_session*>& held);
void sessions_release(std::vector<sv_small_session*>& held);

// Reductions write fixed-order per-block partials into `scratch` and a final
// kernel folds them into `out` (device doubles).
template <typename R>
cudaError_t launch_expect_z_all(const Cx<R>* state, int n, double* scratch, size_t scratch_doubles, double* out,
                                cudaStream_t stream);
template <typename R>
cudaError_t launch_expect_terms(const Cx<R>* state, int n, const sv_pauli_term* terms, int n_terms, double* scratch,
                                size_t scratch_doubles, double* out, cudaStream_t stream);
size_t expect_z_all_scratch_doubles(int n);
// The same for `batch` states back to back: out holds batch x (n + 1) doubles.
template <typename R>
cudaError_t launch_expect_z_batch(const Cx<R>* states, int n, int batch, double* scratch, size_t scratch_doubles,
                                  double* out, cudaStream_t stream);
size_t expect_z_batch_scratch_doubles(int n, int batch, size_t amp_bytes);

size_t expect_terms_scratch_doubles(int n, int n_terms);

int device_sm_count();

// Reads and clears the status a pass kernel recorded on the device (SV_OK, or
// SV_ERR_TIMEOUT when a bounded wait ran out); synchronizes `stream`.
int take_sweep_status(cudaStream_t stream);

// ----------------------------------------------------------------- run-time compiled pass kernels
// (sv_jit.cpp).  jit_mode(): 0 off, 1 compile a program structure on its
// second use, 2 on its first (SV_JIT=0 / 1 / 2 in the environment, or
// jit_set_mode; -1 goes back to the environment).
int jit_mode();
void jit_set_mode(int mode);
// The kernel source of one program, empty if the TMA pass would not run it.
template <typename R>
std::string jit_source(const SweepProgram<R>& P);
// Compiled kernels for a circuit's programs (NULL entries: the interpreting
// kernel runs that pass); compiles what the cache lacks, in parallel.
template <typename R>
std::vector<const JitKernel*> jit_compile_programs(const std::vector<SweepProgram<R>>& progs);
// A program's structure key (empty if the TMA pass would not run it): all its
// kernel source is written from, none of its coefficient values.
std::string jit_program_key(const SweepProgram<float>& P);
// The programs' kernels by structure key: counts a use of each key, compiles
// (in the calling thread, in parallel) the keys used at least `threshold`
// times that have no kernel yet; NULL entries interpret.
std::vector<const JitKernel*> jit_program_kernels(const std::vector<SweepProgram<float>>& progs,
                                                  const std::vector<std::string>& keys, int threshold);
// Launches a compiled pass kernel with the interpreting TMA kernel's
// arguments (map: the CUtensorMap, bx: the TmaBoxes).
cudaError_t jit_launch(const JitKernel* k, void* state, const void* map, const void* bx, const void* prog, int ns,
                       int* status, unsigned grid, unsigned block, size_t smem, cudaStream_t stream);
// Generates (and with compile, compiles for sm_<arch>a) every program's kernel
// without a device.
template <typename R>
void jit_check_programs(const std::vector<SweepProgram<R>>& progs, bool compile, int arch, int* n_sources,
                        int* n_compiled, std::string* first_error, std::string* sources);
void jit_stats(long long* compiled, long long* failed, long long* launches, double* compile_seconds,
               std::string* last_error);
bool jit_available(std::string* why);

// Kernel timing (sv_profile_*): Prof p(stream, "sweep", bytes); launch; p.done();
struct Prof {
  Prof(cudaStream_t s, const char* family, double bytes);
  void done();
  cudaStream_t stream;
  const char* family;
  double bytes;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
};

}  // namespace sv
