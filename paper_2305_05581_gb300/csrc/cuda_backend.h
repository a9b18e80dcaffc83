// cuda_backend.h -- CUDA backend of the engine (sm_103a).
#pragma once

#include <cuda_runtime.h>

#include <map>
#include <string>
#include <vector>

#include "engine.h"

namespace tns {

// device memory of the library (devmem.cu): every allocation goes through
// dmalloc / dfree, which count the bytes in use per device and refuse,
// before cudaMalloc, an allocation above the device budget (0: no budget)
cudaError_t dmalloc_raw(void** p, size_t bytes);
template <class T>
inline cudaError_t dmalloc(T** p, size_t bytes) {
  return dmalloc_raw((void**)p, bytes);
}
void dfree(void* p);
struct DevMem {
  long long used = 0, peak = 0, budget = 0;
};
DevMem dmem(int device);
void dmem_set_budget(int device, long long bytes);
void dmem_reset_peak(int device);

struct Tile {  // an output tile of a group: rows [row0, row0+nrows), cols [col0, col0+ncols)
  int g;
  int row0, col0, nrows, ncols;
  int t0, t1;      // task range of this piece (a split tile has several pieces)
  int aside;       // digit kernel: 1 = op(L) and the rows are the side that is contracted with X first, 0 = op(R) and the columns
  long long poff;  // -1: write the output block; else element offset of this piece's partial tile
};

// classes of the FP64 digit kernel (fp64_digits.cu): most rows of the a side
// and columns of the b side of a tile, l and k staged at a time, CTAs per SM
struct DgClass {
  int a, b, km, ctas;
};
constexpr int kDgClasses = 3;
constexpr DgClass kDgClass[kDgClasses] = {{16, 16, 16, 12}, {32, 32, 32, 4}, {64, 56, 32, 2}};
cudaError_t fp64_digits_init();
class CudaBackend;
struct DevList;
struct Tile;
bool prepare_digits(CudaBackend& be, const TaskList& tl, DevList& d, int nvec, long long length);
int digit_vectors(const DevList& d);  // how many vectors the list's images are for
void enqueue_digit_vectors(CudaBackend& be, const DevList& d, const double* xv, long long xs, int nvec, int* failed);
void release_digit_plan(void* plan);
void launch_fp64_digits(int cls, unsigned grid, cudaStream_t s, const void* plan, const Task* tasks,
                        const Group* groups, const Tile* tiles, int tile0, const double* xv, double* yv, long long xs,
                        long long ys, double* part, long long psize, int nv, int* nfailed, int* failed);

struct SplitRed {  // a split tile: sum of nsplit partial tiles (fixed order) -> output
  int g;
  int row0, col0, nrows, ncols;
  int nsplit;
  long long poff;
};

// schedule variants tried by the online autotuner: the split-K target is
// (total cost) / (resident CTAs x SMs x rounds) with rounds = kRounds[v];
// for the tensor-core form variant kWsVariant runs the persistent
// warp-specialised kernel (its own split, rounds 2) instead of one CTA per
// piece; the FP64 form tries the first kFp64Variants
constexpr int kNumVariants = 4;
constexpr double kRounds[kNumVariants] = {1.0, 2.0, 4.0, 2.0};
constexpr int kWsVariant = 3;
constexpr int kFp64Variants = 3;

// one schedule of a work list for the FP64 kernels: tiles split into size
// classes, long task lists cut into partial tiles summed in fixed order
struct FpVariant {
  bool planned = false;
  Tile* tiles = nullptr;
  int ncls[4] = {0, 0, 0, 0};  // tiles per size class (contiguous, class 0 first)
  double ccost[4] = {0, 0, 0, 0};  // estimated FMAs per class (the costliest runs on the launching stream)
  int ntiles = 0;
  SplitRed* reds = nullptr;  // split tiles to reduce after the product kernels
  int nreds = 0;
  int red_el = 0;            // elements of the largest of them
  long long psize = 0;       // partial-tile elements per vector
  double* part = nullptr;    // partial tiles (psize * part_nvec)
  int part_nvec = 0;
  int* failed = nullptr;     // digit classes: how many pieces have no certificate (4 ints), then which
  int failed_nvec = 0;
};

// online autotuner state of one (precision, nvec) use of a work list: the
// first products run the variants in turn and are timed; the fastest is kept
// for the rest of the list's life
struct Tune {
  int step = 0;   // products run so far while tuning
  int best = -1;
  float ms[kNumVariants] = {1e30f, 1e30f, 1e30f, 1e30f};  // fastest sample of each variant
};
// tuning sequence: one untimed product (default variant: first-use effects
// such as cold caches land there), then kTuneRounds timed samples of every
// variant, the fastest sample of each compared
constexpr int kTuneRounds = 2;
// Inside an eigensolver the products feed the next vectors, and a schedule shows
// in the last bits of their partial sums: there the default variant stays unless
// another needs less than this part of its time, so that timing noise does not
// decide where an unconverged solve ends.  FP64 schedules differ by up to 13 %
// and their samples by 1 to 2 %; of the reduced precisions the split reduction's
// speed alone reorders schedules that lie within 20 %.
constexpr double kSteady = 0.8, kSteadyFp64 = 0.97;
constexpr int kDefaultVariant = 1;
inline int pick_variant(const float* ms, int n, double steady) {
  int best = 0;
  for (int i = 1; i < n; ++i)
    if (ms[i] < ms[best]) best = i;
  return ms[best] > steady * ms[kDefaultVariant] ? kDefaultVariant : best;
}
// A digit product takes 0.3 to 0.7 of the FMA kernel's time, and what has no
// certificate is done again by that kernel, in clusters: beyond a fifth the sum
// is no gain.  24 orbitals, D = 512, all sectors: a tenth, 19 against 36 ms; a
// swept step of 16 orbitals with more than a fifth: 14.2 against 13.2 ms.
constexpr double kFailedShare = 0.2;
// Lists below kDigitFlops stay with the FMA kernel: at 8e6 flops digits are no
// faster (12 orbitals, D = 130, 2 sectors: 0.066 and 0.075 ms), at 2.6e7 they are
// (8 orbitals: 0.235 and 0.177 ms).  Making the images takes a product 0.2 ms,
// more than the first product gains below kDigitsAtOnce (8 orbitals 1.36 -> 1.60
// ms, 10 orbitals at 9.4e7 flops 2.40 -> 2.62; at 4.4e8 and above the same or
// less): there they are made with the second one.
constexpr double kDigitFlops = 2e7, kDigitsAtOnce = 4e8;
constexpr int kSteadyKey = 1 << 16;  // schedules and graphs of such products are kept apart

// captured launch sequence of one (precision, nvec) use: replayed with the
// input copied into xbuf and the output copied out of ybuf
struct GraphSlot {
  cudaGraphExec_t exec = nullptr;
  double* xbuf = nullptr;
  double* ybuf = nullptr;
  long long elems = 0;  // doubles per buffer (nvec * stride)
  long long stride = 0;
  int kernels = 0;      // kernel launches inside the graph
  bool failed = false;  // capture not possible: launch directly
};

// device copy of a work list
struct DevList {
  long long gen = -1;
  unsigned long long shape = 0;  // shape signature of the list (schedule cache key)
  Task* tasks = nullptr;
  Group* groups = nullptr;
  Tile* wtiles = nullptr;    // 32 x 16 warp tiles of the FP64 tensor (DMMA) kernel
  int nwtiles = 0;
  FpVariant fv[2][kNumVariants];  // [0] DFMA classes, [1] digit classes
  // FP64 output tiles per size class with their estimated FMAs (host; shared
  // by the schedule variants, which differ only in how they cut the tiles)
  bool fp_tiled[2] = {false, false};
  std::vector<Tile> fp_tiles[2][4];
  std::vector<double> fp_cost[2][4];
  // digit images of the list (fp64_digits.cu); dg_none: they cannot be had
  void* dg = nullptr;
  bool dg_none = false;
  double flops = -1;     // of the list's products, once asked for
  bool dg_kept = false;  // the first product's certificates held (kFailedShare)
  std::vector<unsigned char> dg_aside;  // per group: the tiles' a side
  // tensor-core form (precision != FP64)
  void* tc = nullptr;
  long long tc_gen = -1;
  std::map<int, Tune> tune;         // key: precision code * 64 + nvec (+ kSteadyKey)
  std::map<int, GraphSlot> graphs;  // same key
};

class CudaBackend : public Backend {
 public:
  CudaBackend(int device, cudaStream_t s, bool own);
  // FP64 product kernel of every list: 0 DFMA tile classes, 1 DMMA (mma.sync
  // m8n8k4 f64), 2 exact digit products on the f16 tensor cores
  // (fp64_digits.cu) where a list has images; -1 (default): digits where the
  // list allows them, else DFMA; environment TNS_FP64_KERNEL=dfma|dmma|digits
  int fp64_kernel = -1;
  // bound of one wait inside the tensor-core product loop (ns); the
  // environment variable TNS_TC_WAIT_NS overrides the default 0.2 s when the
  // backend is created (a test makes the waits run out with it and checks the
  // reported error and that the context stays usable; with 0 every CTA of the
  // tile kernel and every warp of the small-block kernel first waits on a
  // barrier that nothing completes, since its copies may land before any wait
  // could run out)
  unsigned long long tc_wait_ns = 200000000ull;
  // TNS_TC_VARIANT=v (0..kNumVariants-1) fixes the tensor-core schedule
  // variant instead of tuning it (tests run each kernel this way)
  int forced_tc_variant = -1;
  // output blocks whose dimensions, and those of every X block they read, are
  // at most tc_small go to the warp-level small-block kernel of the
  // tensor-core form (0: every block to the tile kernel; at most 32);
  // environment TNS_TC_SMALL
  int tc_small = 32;
  // destroy the CUDA graphs captured for a work list (after both streams
  // have drained): every buffer a graph reads or writes is baked into it, so
  // they go before any such buffer is freed or reallocated
  void free_graphs(DevList& d);
  ~CudaBackend() override;
  double* alloc(long long n) override;
  void release(double* p) override;
  void upload(double* dst, const double* src, long long n) override;
  void download(double* dst, const double* src, long long n) override;
  void zero(double* p, long long n) override;
  void copy(double* dst, const double* src, long long n) override;
  bool trim() override;
  void lincomb(const LCList& l) override;
  void run(const TaskList& tl, const double* xv, double* yv, int nvec, long long xs, long long ys,
           int precision) override;
  void task_values(const TaskList& tl, const double* xv, const double* ybar, double* out) override;
  void nonzero_blocks(const std::vector<const double*>& p, const std::vector<long long>& n,
                      std::vector<char>& nz) override;
  long long mem_used() override;
  long long mem_limit() override;
  long long mem_free() override;
  void set_budget(long long bytes) override;
  double* host_alloc(long long n) override;
  void host_release(double* p) override;
  void forget(const TaskList& tl) override { drop(tl); }
  long long step_bytes(const TaskList& tl, long long psi_length) override;
  void sync() override;
  std::string error() override;

  cudaStream_t stream() const { return stream_; }
  int device() const { return device_; }
  void note(cudaError_t e, const char* what);
  // false once a failure (an allocation, a launch) has been noted in the
  // current call: later launches are skipped so that no kernel runs on a
  // buffer that does not exist
  bool ok() const { return err_.empty(); }
  // persistent device copy of a task list (uploaded when tl.gen changes)
  DevList& dev(const TaskList& tl);
  // the device copy of tl if it is resident and current, else nullptr (never uploads)
  const DevList* resident(const TaskList& tl) const {
    auto it = lists_.find(&tl);
    return (it != lists_.end() && it->second.gen == tl.gen && it->second.tasks) ? &it->second : nullptr;
  }
  void drop(const TaskList& tl);
  // CUDA graphs for persistent work lists (on by default; TNS_GRAPHS=0 turns
  // them off)
  bool use_graphs = true;
  // online schedule autotuning (on by default; TNS_AUTOTUNE=0 keeps the
  // default variant, which makes repeated runs bitwise reproducible)
  bool autotune = true;
  // device bytes the last step's memory plan asked for (step_bytes)
  long long last_step_bytes = 0;
  bool iterating = false;  // products of an eigensolver (kSteady)
  // launches of the FP64 product kernels of variant v (no allocation, no
  // synchronisation: capturable)
  void enqueue_fp64(const DevList& d, int dig, int v, const double* xv, double* yv, int nvec, long long xs, long long ys);
  void enqueue_fp64_vectors(const DevList& d, int dig, const FpVariant& f, const double* xv, double* yv, int nvec,
                            long long xs, long long ys, double* part);
  // room for `bytes` of the backend's own allocations (the engine's hook)
  void need(long long bytes) {
    if (room && bytes > (64LL << 20)) room(bytes);
  }
  // scratch device memory owned by the backend (grows, never shrinks)
  void* scratch(size_t bytes, int slot);
  // counted launches of the engine's own kernels
  long long launches = 0;
  // schedule tuning: lists tuned, lists that took a cached choice, and how
  // often each variant ran as the chosen one (per precision: 0 FP64, 1 TF32, 2 BF16X3)
  long long tuned = 0, tune_cache_hits = 0;
  long long variant_runs[3][kNumVariants] = {};
  float last_ms = 0.f;

 private:
  int device_;
  int sms_ = 152;
  cudaStream_t stream_;
  bool own_;
  std::string err_;
  std::map<const TaskList*, DevList> lists_;
  const DevList* running_ = nullptr;  // the list of the current run()
  // best schedule variant per (precision, nvec, shape signature): work lists
  // of later steps with the same shape take it without tuning again
  std::map<std::pair<int, unsigned long long>, int> tune_cache_;
  std::vector<std::pair<void*, size_t>> scratch_ = std::vector<std::pair<void*, size_t>>(8, {nullptr, 0});
  cudaStream_t gstream_ = nullptr;  // side stream for graph capture and replay
  cudaEvent_t gev_[2] = {nullptr, nullptr};
  // forked streams: the FP64 tile classes run side by side (fork/join events)
  cudaStream_t fstream_[3] = {nullptr, nullptr, nullptr};
  cudaEvent_t fev_[4] = {nullptr, nullptr, nullptr, nullptr};
  bool fork_ready();
  double failed_share(const FpVariant& f, int nvec);
  void upload_list(const TaskList& tl, DevList& d);
  void plan_variant(const TaskList& tl, DevList& d, int dig, int v);
  bool ensure_part(DevList& d, FpVariant& f, int dig, int nvec);
  void free_list(DevList& d);
  template <class F>
  void launch_graphed(DevList& d, int key, const double* xv, double* yv, int nvec, long long xs, long long ys,
                      F&& enqueue);
};

// allocation-free H_eff diagonal (noalloc.cu)
int heff_diag_noalloc(CudaBackend& be, Step& st, double* diag, std::string& err);

// tensor-core form (tc.cu): prepare (plan, allocations; not capturable),
// enqueue (kernel launches only; capturable), check (reads the timeout flag,
// synchronises)
bool prepare_tasks_tc(CudaBackend& be, const TaskList& tl, DevList& d, int nvec, int variant, int precision);
void enqueue_tasks_tc(CudaBackend& be, DevList& d, const double* xv, double* yv, int nvec, long long xs,
                      long long ys, int precision, int variant);
void check_tasks_tc(CudaBackend& be, DevList& d);
void release_tc_plan(void* plan);

// kernels used by the solver (defined in kernels.cu)
void launch_reduce_splits(CudaBackend& be, const SplitRed* reds, int nreds, int maxel, const Group* groups,
                          const double* part, long long psize, double* yv, long long ys, int nvec);
void launch_heff_diag(CudaBackend& be, const Task* d_tasks, const int* d_idx, const int* d_rng, int ngroups,
                      const Group* d_groups, double* diag);
void launch_multidot(CudaBackend& be, const double* V, long long ldv, int k, const double* w, long long n,
                     double* out);
void launch_axpy_multi(CudaBackend& be, const double* V, long long ldv, int k, const double* coef, double sign,
                       double* w, long long n);
void launch_combine(CudaBackend& be, const double* V, long long ldv, int k, const double* coef, double* out,
                    long long n);
void launch_scale(CudaBackend& be, double* x, const double* num, int inv_sqrt, long long n);
void launch_precond(CudaBackend& be, const double* r, const double* diag, const double* theta, double* t,
                    long long n);
void launch_residual(CudaBackend& be, const double* AVs, const double* x, const double* theta, double* r,
                     long long n);
// batched symmetric eigensolver (cyclic Jacobi), matrices column-major == row-major (symmetric)
// A: nmat matrices at A + off[i] with size n[i]; V: eigenvectors (columns) at V + off[i]; w: eigenvalues at w + woff[i]
void launch_jacobi(CudaBackend& be, double* A, double* V, double* w, const long long* off, const int* n,
                   const int* woff, int nmat, int maxn, int* sweeps_out);
// batched symmetric eigensolver (Householder tridiagonalisation + implicit QR),
// one CTA per matrix; eigenvector p is ROW p of Z (Z + off[i], n x n); A is
// overwritten; *status (nullable) is set to 1 if a matrix hit the QR step limit
constexpr int SYEV_MAXN = 4096;
void launch_syev(CudaBackend& be, double* A, double* Z, double* w, const long long* off, const int* n,
                 const int* woff, int nmat, int maxn, int* status);
void launch_select(CudaBackend& be, const double* w, const int* sec_of, int total, int keep_max, double cut,
                   int* keep_flag, double* disc);
void launch_gather(CudaBackend& be, const double* src, const long long* so, const int* sld, double* dst,
                   const long long* dof, const int* dld, const int* rows, const int* cols, const int* trans,
                   int nblk);
void launch_argmin(CudaBackend& be, const double* x, long long n, long long* idx);
void launch_fill_unit(CudaBackend& be, double* x, long long n, const long long* idx);

}  // namespace tns
