// pc_handles.h -- the opaque handles of include/pc.h and the host helpers
// shared by the entry-point files (pc_capi.cpp, pc_batch.cpp).  Private to
// the library.
#pragma once

#include <cstdint>
#include <map>
#include <mutex>
#include <set>
#include <string>
#include <utility>
#include <vector>

#include <cuda_runtime.h>

#include "pc.h"
#include "pc_internal.h"

// A run-time specialised pricing kernel: the program it was compiled from
// (code and pool words), the underlying count and the per-path variant.
// Kinds of run-time specialised kernels: pricing (bit kJitPriceWrite: with
// per-path payoffs; bit kJitHbm: the window of dates in HBM; bit
// kJitWinRegs: a window of one date, kept in registers; bit kJitPairs2 (with
// kJitWinRegs): four paths a lane), and the
// control-variate kernel (kJitCv + its kCv* mode bits), the tangent kernel
// (kJitGreeks, + 1: per-path outputs) and the adjoint kernel (kJitAdjoint,
// + 1: per-path outputs).
constexpr int kJitPrice = 0, kJitPriceWrite = 1, kJitHbm = 2, kJitWinRegs = 4, kJitPairs2 = 8, kJitCv = 16,
              kJitGreeks = 32, kJitAdjoint = 64;
// resident blocks per SM the specialised pricing kernel's register bound is
// set for by default (<= 72 registers at 128 threads: the fastest measured)
constexpr int kJitMinBlocks = 7;
// one underlying needs fewer registers: 8 blocks (<= 64).  Averages over 20,
// 35 and 60 dates and barriers over 20 to 60, us at 7 / 8 blocks: 3e5 paths,
// where 7 leave a second round, 38.9 / 27.0, 58.6 / 40.8, 94.8 / 63.6 and
// 35.0 / 24.7 to 77.9 / 53.4; 5e5 and 1e6 paths up to 7 % faster (20 dates,
// 5e5: 43.8 / 44.1); 2^14 to 1.5e5 within 3 %, most equal (20 dates, 5e4: 21.3
// / 22.6).  Four paths a lane (100 and 252 dates): within 2 %, 4 % faster at 1e6.
constexpr int kJitMinBlocks1 = 8;
// the same with a static walk, whose bridge stack and normals are registers
// (autocall, 3 underlyings, 5 dates, 2^20 paths: 5 / 6 / 7 / 8 blocks 52.5 / 51.4 / 52.1 / 52.1 us a call)
constexpr int kWalkMinBlocks = 6;
// resident blocks per SM the specialised control-variate kernel's register bound is set for
constexpr int kJitCvMinBlocks = 5;
// dates of the model from which a one-date-window kernel takes two path pairs a lane
constexpr int kJitPairsMinDates = 64;
constexpr size_t kJitStaticSmem = 256;  // bound on price_tiles' static shared memory

// What a specialised kernel is compiled for beside its program.
struct JitSpec {
  int d = 0;
  int kind = kJitPrice;
  int min_blocks = 0;  // its launch bound's resident blocks per SM (0: the kernel's own)
  // a static walk over the dates that the program reads (see static_walk in
  // pc_capi.cpp): per step the date, 1 if it is read, the number of bridge
  // ops and their numbers; empty: the general walk
  std::vector<int32_t> walk;
  // the launch's layout as constants (empty, or a field of -1: read from the
  // arguments; see jit_spec) and with a walk the model's n, n_hist and t_now
  std::vector<int32_t> lay, grid;
  bool one_phi = false;  // every path of the launch has the same upper 32 index bits
  bool operator==(const JitSpec &o) const {
    return d == o.d && kind == o.kind && min_blocks == o.min_blocks && one_phi == o.one_phi && walk == o.walk &&
           lay == o.lay && grid == o.grid;
  }
};

struct JitEntry {
  std::vector<uint32_t> program;
  JitSpec spec;
  cudaLibrary_t lib = nullptr;
  cudaKernel_t kernel = nullptr;
};

// Device scratch, grown on demand (grow_scratch) and shared by the calls.
struct Scratch {
  void *p = nullptr;
  size_t bytes = 0;
  bool captured = false;  // a caller's graph holds the address
  template <typename T>
  T *as() const { return static_cast<T *>(p); }
};

struct pc_ctx {
  int device = 0;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  int sm_count = 0;
  int max_smem = 0;
  int sm_smem = 0;       // shared memory per SM (bytes)
  int smem_reserve = 0;  // shared memory the system reserves per resident block (bytes)
  double *d_res = nullptr;       // [8]: sum, sumsq, n, -, status word (int32 at d_res+4)
  double *d_gout = nullptr;      // [PC_MAX_UNDERLYINGS * 8]: sensitivity sums per underlying
  Scratch partials;              // tile partials (doubles)
  unsigned char *d_control = nullptr;  // reduction control block (kControlBytes, zero between launches)
  Scratch tape;                  // adjoint tapes, one region per resident warp
  Scratch gwin;                  // HBM windows of simulated dates (float2 slots)
  Scratch screen;                // screened launches: count, list and payoffs (4-byte words)
  std::vector<void *> captured;  // scratch that grew after a caller's graph took its address: kept until the context goes
  int32_t window_mode = 0;       // PC_WINDOW_AUTO / _SHARED / _HBM
  int32_t jit = 0;               // 1: price with run-time specialised kernels
  // streams and events of one-shot portfolio launches (pc_price_batch),
  // created once per context
  std::vector<cudaStream_t> batch_aux;
  std::vector<cudaEvent_t> batch_join;
  cudaEvent_t batch_fork = nullptr;
  int32_t cv_min_blocks = 0;     // launch bound of the specialised control-variate kernel (0: its default)
  int32_t jit_pairs = 0;         // path pairs a lane of a specialised kernel with a one-date window (0 automatic, 1 or 2)
  std::mutex jit_mu;
  std::multimap<uint64_t, JitEntry> jit_cache;  // program hash -> compiled kernels
  std::map<uint64_t, std::vector<std::vector<int32_t>>> jit_walks;  // program hash -> its static walks (admit_walk)
  std::map<std::pair<const void *, size_t>, int> jit_occ;  // (kernel, smem) -> resident blocks
  std::map<const void *, size_t> jit_smem;                 // kernel -> the most dynamic shared memory it was set for
  cudaMemPool_t pool = nullptr;  // stream-ordered allocations of contracts (null: cudaMalloc)
  double *h_res = nullptr;       // pinned [64]: the blocking calls' results, written by the kernel
  uint64_t *h_done = nullptr;    // pinned: (ticket << 32) | device status, written after them
  uint32_t ticket = 0;           // the last blocking call's
  // pinned staging of program uploads, two halves filled in turn: a half is
  // reused once the event recorded when it was left has completed
  uint32_t *h_stage = nullptr;
  size_t stage_words = 0;        // words per half
  size_t stage_off = 0;          // next free word in the current half
  int stage_half = 0;
  cudaEvent_t stage_ev[2] = {nullptr, nullptr};
  bool stage_pending[2] = {false, false};
  // compiled programs by their inputs (bytecode, constants, template
  // parameters, parties): reloading a program skips the compiler
  std::mutex load_mu;
  std::multimap<uint64_t, std::pair<std::vector<uint32_t>, pc::Program>> program_cache;
  double timeout_s = 300.0;
  int32_t fail_allocs = 0;       // failure injection: this many next allocations fail (pc_debug_fail_allocations)
  int live_objects = 0;
};

struct pc_contract;

struct pc_model {
  pc_ctx *ctx = nullptr;
  pc::ModelHost H;
  void *d_mem = nullptr;
  pc::ModelDev dev{};
  uint64_t id = 0;
  mutable std::set<pc_contract *> users;  // contracts that keep a Window of this model
};


struct pc_contract {
  pc_ctx *ctx = nullptr;
  pc::Program prog;
  pc::XInsn *d_code = nullptr;
  bool pooled = false;            // d_code came from the context's memory pool
  std::vector<uint32_t> image;    // program then padded pool: the uploaded words
  std::mutex mu;
  // (an entry goes with its model: pc_model_destroy)
  struct Window {
    const pc_model *model = nullptr;
    int32_t win = 1, skip = 0;
    bool with_walks = false;  // computed for specialised kernels
    // static walks over the dates the program reads, and over every date
    // of the model (a per-date hook); empty where they are too long; and
    // their launch arguments
    std::vector<int32_t> walk, walk_all;
    pc::StaticGrid grid{}, grid_all{};
    // the specialised kernels found for this pair so far (jit_kernel's
    // answers: looking one up by its program costs a microsecond or two)
    struct Kernel {
      int kind, min_blocks, words;
      bool one_phi;
      cudaKernel_t kernel;
    };
    std::vector<Kernel> kernels;
  };
  std::map<uint64_t, Window> win_cache;  // by model id
};

namespace pc {

// Device memory on the context's stream: from its memory pool (stream
// ordered, no device synchronisation) when it has one, else cudaMalloc.
cudaError_t ctx_alloc(pc_ctx *c, void **p, size_t bytes, bool &pooled);
void ctx_free(pc_ctx *c, void *p, bool pooled);
// Resident blocks per SM of a run-time compiled kernel at this dynamic
// shared memory (sets its shared-memory limit on first use; memoised).
cudaError_t jit_occupancy(pc_ctx *c, const void *kern, int block, size_t smem, int &blocks);

// Record a message for pc_last_error and return the status.
pc_status fail(pc_status s, const std::string &m);
pc_status cuda_fail(cudaError_t e, const char *what);

#define CU(call, what)                                 \
  do {                                                 \
    cudaError_t e_ = (call);                           \
    if (e_ != cudaSuccess) return ::pc::cuda_fail(e_, what); \
  } while (0)

// Wait for the context's stream with its wall-clock limit.
pc_status wait_stream(pc_ctx *c);

// A blocking call's results: the launch writes its sums to pinned host memory
// and then the call's ticket with the device status to a pinned word, which
// the host polls (with the wall-clock limit; the stream is queried now and
// then, for errors).  A copy back and a stream query took 4 us more, two
// copies to pageable memory 15.
void report_to_host(pc_ctx *c, PriceArgs &a);       // sets a.done and a.ticket (the call's last launch)
pc_status wait_report(pc_ctx *c);                   // results in c->h_res; PC_EDEVICE for a raised status

// cudaMalloc for the context's buffers, or a simulated out-of-memory
// (cudaErrorMemoryAllocation, nothing allocated) while the context's
// failure injection count is positive.
cudaError_t ctx_malloc(pc_ctx *c, void **p, size_t bytes);

// Room left for a kernel's static shared memory when sizing its dynamic
// shared memory.
constexpr size_t kStaticSmemReserve = 2048;

// Constant-pool floats of a program, rounded up to whole 16-byte words.
size_t pool_padded(const Program &p);

// A pricing launch: per-contract arguments plus its single-launch shape.
struct Launch {
  PriceArgs args{};
  int grid = 0;
  int block = kBlock;
  size_t smem = 0;
  pc_contract::Window *w = nullptr;  // the contract on the model: its static walks and kernels
  bool hbm_window = false;  // window in HBM (args.lay.gwin set by the launcher)
  int sparse_grid = 0;      // the dense variant's launch (PriceKind): the grid without it, else 0
};

// Validate (model, contract, n_paths), resolve the contract's date window for
// the model and fill the per-contract arguments (everything but the
// reduction scratch and outputs) and a single-launch shape.  With
// allow_hbm the window may be placed in HBM (pricing kernel only): when the
// context asks for it, or (automatic mode) when the shared window would
// leave fewer than 8 resident warps per SM or exceeds PC_MAX_WINDOW.
// specialised: for a specialised kernel although the context interprets.
pc_status prepare(const pc_model *m, const pc_contract *k, uint64_t n_paths, uint64_t offset,
                  uint64_t seed, uint32_t stream, Launch &L, bool allow_hbm = false, bool specialised = false);

// Whether the caller is capturing the context's stream.
bool capturing(const pc_ctx *c);
// A scratch buffer of at least `bytes`.  Under a caller's capture its address
// goes into the caller's graph: nothing is grown then (PC_ECUDA, the capture
// unharmed), and when the buffer grows later the captured one is kept until
// the context goes, so that the graph may be replayed after any call.
pc_status grow_scratch(pc_ctx *c, Scratch &b, size_t bytes, const char *what);
// The context's tile-partial scratch for at least `doubles`.
pc_status ensure_partials(pc_ctx *c, size_t doubles);

// The run-time specialised kernel of the contract's program for d
// underlyings, a kernel kind (kJit*), a register bound and a walk; compiled
// on first use, cached on the context by program content.
pc_status jit_kernel(const pc_contract *k, const JitSpec &spec, cudaKernel_t &out);
// Programs of at most PC_JIT_MAX_INSNS instructions are specialised; the
// launches of longer ones interpret them.
bool jit_eligible(const pc_contract *k);
// A program the specialised adjoint kernel takes: one of at most
// kAdjointDateSites reading instructions (pc_jit.cpp).
bool adjoint_jit_eligible(const pc_contract *k);
// A program whose evaluator can take a static walk: one copy of it, or two.
bool walk_jit_eligible(const pc::Program &p);
// A static walk's kernel is compiled for the grid too, so a program priced on
// models of ever new grids would compile each time: whether this walk on this
// model is one of the context's first kWalksPerProgram of the program (the
// others take the general kernel, compiled once).
constexpr size_t kWalksPerProgram = 8;
bool admit_walk(pc_ctx *c, const Program &p, const ModelHost &H, const std::vector<int32_t> &walk);
// The launch argument of a static walk on a model.
StaticGrid static_grid(const ModelHost &H, const std::vector<int32_t> &walk);
// Whether every path of offset .. offset + n_tiles tiles has the same p_hi.
inline bool one_phi(uint64_t offset, uint64_t n_tiles) {
  return (offset >> 32) == ((offset + n_tiles * kTilePaths - 1) >> 32);
}
// Compile the specialised kernels of many requests into the context's cache
// (those not there yet), NVRTC on the host's cores in parallel; jit_kernel
// then finds them.
struct JitRequest {
  const pc_contract *k;
  JitSpec spec;
};
pc_status jit_compile_many(pc_ctx *c, const std::vector<JitRequest> &reqs);
// The specialised pricing kernel's variant for a prepared launch (window in
// registers, path pairs a lane, HBM window), its layout (the launch's shared
// memory; may re-choose the block) and the register bound it is compiled for.
int jit_window_kind(const pc_ctx *c, const Launch &L);
size_t jit_layout(const pc_ctx *c, Launch &L, int bits);
int jit_min_blocks(const pc_ctx *c, size_t smem, int block, int d);
// What the contract's specialised kernel of `kind` is compiled for: the
// launch's arguments (layout final) and a walk (may be empty).
JitSpec jit_spec(const pc_contract *k, const PriceArgs &a, int kind, int min_blocks, const std::vector<int32_t> &walk);
JitSpec jit_price_spec(const pc_ctx *c, const pc_contract *k, const Launch &L, int kind, size_t smem);
// jit_kernel of jit_spec, or the pair's earlier answer for the same launch.
pc_status jit_pair_kernel(const pc_contract *k, pc_contract::Window *w, const PriceArgs &a, int kind, int min_blocks,
                          const std::vector<int32_t> &walk, cudaKernel_t &out);
void drop_bridge_stack(Layout &lay);
void jit_release(pc_ctx *c);

// Turn a raised device status word into PC_EDEVICE (and clear it).
pc_status check_status(pc_ctx *c, int32_t status);

}  // namespace pc
