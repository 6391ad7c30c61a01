// Library state shared by the host API and the CUDA kernels.
#pragma once
#include <cuda_runtime.h>

#include <string>
#include <vector>

#include "su2_internal.h"

// FP64 products: 64x64 output tiles.
namespace su2 {
constexpr int kTile = 64;

// ---- FP64 H.psi: stacked products (heff_fp64.cu)
// K1: the T(k1 x n) = E(k1 x k2) . D(n x k2)^T of one input block and all the
// right operator blocks its tasks read, side by side
struct P64Ent { int64_t d_off, t_off; int32_t n, col0; };  // one right block: its columns start at col0
struct P64In { int64_t e_off; int32_t k1, k2, ent0, ent1, ncol, pad; };
struct P64K1 { int32_t in, ent, tr, tc; };                 // one tile; ent: the entry that holds its first column
// K2: F of all output blocks with one left sector (contiguous in psi: m x N)
// += [A_1 A_2 ..] [T'_1; T'_2; ..], T'(w, f) = sum_t v_t T_t over the tasks of
// left block w and output block f
struct P64Left { int64_t a_off; int32_t k0, pad; };        // A block (-1: identity), its first K
struct P64Task { int64_t off; double v; int32_t ld, psi; };
struct P64Col { int32_t f, c; };
struct P64Stack { int64_t f_off, tab_off; int32_t left0, step0, nf, N, m, K, col0, pad; };
struct P64K2 { int64_t part; int32_t st, tr, tc, s0, s1, pad; };  // K steps [s0, s1) of one tile; part >= 0: a partial tile, stored there
struct P64Tile { int64_t f_off, part0; int32_t rows, cols, ld, npart; };  // npart partial tiles (rows x cols, no padding) from part0
struct Chunk64 {
  int64_t k1_begin, k1_end, k2_begin, k2_end, sp_begin, sp_end;
  double k1_flops, k2_flops;
};
struct Plan64 {
  std::vector<Chunk64> chunks;
  std::vector<P64Ent> ent;
  std::vector<P64In> in;
  std::vector<P64K1> k1;
  std::vector<P64Left> left;
  std::vector<int32_t> step, tab;
  std::vector<P64Task> task;
  std::vector<P64Col> col;
  std::vector<P64Stack> stack;
  std::vector<P64K2> k2;
  std::vector<P64Tile> tile;
  int64_t n_part = 0;  // doubles of a chunk's partial tiles (the most of any chunk; behind T in the environment's dT)
  P64Ent* d_ent = nullptr;
  P64In* d_in = nullptr;
  P64K1* d_k1 = nullptr;
  P64Left* d_left = nullptr;
  int32_t *d_step = nullptr, *d_tab = nullptr;
  P64Task* d_task = nullptr;
  P64Col* d_col = nullptr;
  P64Stack* d_stack = nullptr;
  P64K2* d_k2 = nullptr;
  P64Tile* d_tile = nullptr;
  double* d_part = nullptr;
};

// ---- FP64 products of the renormalisation (renorm.cu)
// K1: T(k1 x n) = E(k1 x k2) . D(n x k2)^T for one deduplicated
// (right operator block, input block) pair, one 64x64 tile of T.
struct K1Job {
  int64_t e_off, d_off, t_off;
  int32_t k1, k2, n, tr, tc, pad;
};
// K2: one 64x64 tile of an output block F{f}, summed over the tasks
// [t0, t1) of the current chunk that write into f (output stationary).
struct K2Job {
  int64_t f_off;
  int32_t m, n, tr, tc, t0, t1;
  int64_t part;  // >= 0: a run of the tile's tasks, stored there as a partial tile
};
struct K2Task {
  int64_t a_off;  // left operand (m x k1)
  int64_t b_off;  // T in the chunk buffer (k1 x n)
  int32_t k1, pad;
  double v;       // coefficient
};
struct DiagJob {  // one 64 x 64 tile of a block of the diagonal, its diagonal tasks [t0, t1)
  int64_t f_off;
  int32_t m, n, tr, tc, t0, t1;
};
struct DiagTask {
  int64_t a_off, d_off;  // -1: identity
  int32_t lda, ldd;
  double v;
};
struct Chunk {
  int64_t k1_begin, k1_end, k2_begin, k2_end, sp_begin, sp_end;
  double k1_flops, k2_flops;
};

// CUDA-event profiling of the hot-path launches
constexpr int kProfKinds = 6;  // kind 5 counts every hot-path kernel launch
struct Profiler {
  bool on = false;
  struct Pending { int kind; cudaEvent_t a, b; double flops; };
  std::vector<Pending> pending;
  std::vector<cudaEvent_t> pool;
  int64_t launches[kProfKinds] = {};
  double ms[kProfKinds] = {};
  double flops[kProfKinds] = {};
  cudaEvent_t get() {
    cudaEvent_t e;
    if (!pool.empty()) { e = pool.back(); pool.pop_back(); }
    else cudaEventCreate(&e);
    return e;
  }
  // returns the pending slot; call end() after the launch
  void count(int n) { launches[5] += n; }
  int begin(cudaStream_t s, int kind, double fl) {
    if (!on) return -1;
    Pending p{kind, get(), get(), fl};
    cudaEventRecord(p.a, s);
    pending.push_back(p);
    return int(pending.size()) - 1;
  }
  void end(cudaStream_t s, int slot) {
    if (slot >= 0) cudaEventRecord(pending[slot].b, s);
  }
  void drain() {
    for (auto& p : pending) {
      cudaEventSynchronize(p.b);
      float t = 0.f;
      cudaEventElapsedTime(&t, p.a, p.b);
      ms[p.kind] += t;
      launches[p.kind] += 1;
      flops[p.kind] += p.flops;
      pool.push_back(p.a);
      pool.push_back(p.b);
    }
    pending.clear();
  }
  void reset() {
    drain();
    for (int i = 0; i < kProfKinds; ++i) { launches[i] = 0; ms[i] = 0; flops[i] = 0; }
  }
  ~Profiler() {
    for (auto& p : pending) { cudaEventDestroy(p.a); cudaEventDestroy(p.b); }
    for (auto e : pool) cudaEventDestroy(e);
  }
};

// tasks whose four dimensions are all at most kSmallDim run in FP64 on CUDA
// cores in the split path (the small-task class)
constexpr int kSmallDim = 16;

// one chunk of the renormalisation's products (split: its tiles with several K2 jobs)
void launch_heff_fp64(cudaStream_t s, const double* L, const double* R, const double* psi, double* F, double* T,
                      const K1Job* k1, const K2Job* k2, const K2Task* tasks, const P64Tile* split, double* part,
                      const Chunk& c);
// one term chunk of the FP64 H.psi: F += its terms (T: the chunk's intermediates)
void launch_stack_fp64(cudaStream_t s, const Plan64& p, const Chunk64& c, const double* L, const double* R,
                       const double* psi, double* F, double* T, Profiler* prof);
void launch_diag(cudaStream_t s, const double* L, const double* R, double* d, const DiagJob* jobs, int64_t njobs,
                 const DiagTask* tasks, int64_t psi_len);
}  // namespace su2

namespace su2 {
// Out-of-core operator arenas (Sec. III.E-F).  The operator blocks of both
// sides share one logical arena laid out by the planner: [0, prefix) is
// resident on the device (blocks shared by several term chunks, blocks of
// the diagonal and of the small-task class, then the blocks of the first
// chunks up to the device budget), the rest lies in pinned host memory with
// the blocks of each chunk contiguous, [hs[c], he[c]).  Per H.psi the
// streamed range of chunk c is copied on a dedicated IO stream into device
// slot c % 2 while other chunks compute; events order each copy after the
// last reader of its slot and each chunk after its copy.
struct OpStream {
  bool on = false;
  std::vector<int> starts;       // term chunk boundaries (shared by the FP64 and split plans)
  int64_t prefix = 0;            // doubles resident on the device
  int64_t total = 0;             // doubles of the logical arena
  std::vector<int64_t> hs, he;   // streamed range of each chunk (logical offsets)
  int64_t slot = 0;              // doubles per device slot
  int64_t t64 = 0;               // bytes of the largest chunk's T on the FP64 path
  int64_t work = 0;              // bytes of the intermediates of the largest chunk (either path, up to kMaxSlices slices)
  double* dbuf = nullptr;        // device: [0, prefix) resident, then the two slots
  double* host = nullptr;        // pinned host memory: logical [prefix, total)
  cudaStream_t io = nullptr;
  cudaEvent_t copied[2] = {nullptr, nullptr}, freed[2] = {nullptr, nullptr};
  cudaEvent_t fork = nullptr, join = nullptr;
  double io_bytes = 0.0;         // bytes copied per H.psi
  // the diagonals of the blocks the diagonal of H_eff reads (device, kept):
  // block b of side sd has its diagonal at ddiag[dg_off[sd][b]] (-1: none)
  std::vector<int64_t> dg_off[2];
  int64_t dg_total = 0;
  double* ddiag = nullptr;
  // device offset of a block at logical offset `off` read by chunk c
  int64_t dev_off(int64_t off, int c) const {
    return off < prefix ? off : prefix + int64_t(c & 1) * slot + (off - hs[size_t(c)]);
  }
};
}  // namespace su2

namespace su2 {
// ---- sizes of the split path's stacks (heff_split.cu), shared with the out-of-core planner
constexpr int kMaxSlices = 6;
// left blocks that are the block Hamiltonian: the left operators of the terms
// that act on nothing else
std::vector<char> left_hamiltonians(const OpTable& t);
// K axis of the stacked left blocks of one output sector: 16-K steps of an
// exponent group, steps of the whole, first 8-K piece of each block (and the
// end).  own: the block begins and ends a group
struct StackK { int gst = 0, kst = 0; std::vector<int> at; };
StackK stack_k(const std::vector<int>& cols, const std::vector<char>& own);
}  // namespace su2

struct su2_ctx {
  int device = -1;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  std::string err;
  int* d_status = nullptr;
};

struct su2_sectors {
  int site_kind = 0, N = 0, twoS = 0;
  std::vector<su2::Sector> left, right;
  std::vector<su2::Block> blocks;
  std::vector<su2_block> pub;
  int64_t psi_len = 0;
};

struct su2_env {
  su2_ctx* ctx = nullptr;
  int device = -1;  // the context's device, kept here so that destroying the
                    // environment never reads its context (which the caller
                    // may already have destroyed)
  su2::OpTable table;
  su2::SideOps L, R;
  std::vector<su2::Task> tasks;
  su2_env_info info{};
  int64_t psi_len = 0;
  std::vector<su2::Block> blocks;   // psi blocks
  std::vector<su2::Sector> lsec, rsec;
  int64_t split_budget = 0;
  int spin_limit = 0;  // polls of each work-loop wait of the split GEMM (0: the kernel's default)
  su2::Plan64 p64;  // FP64 plan
  std::vector<su2::DiagJob> dj;
  std::vector<su2::DiagTask> dt;
  int64_t t_elems = 0;  // T buffer size (doubles)
  // device copies
  double *dL = nullptr, *dR = nullptr, *dT = nullptr;
  su2::DiagJob* ddj = nullptr;
  su2::DiagTask* ddt = nullptr;
  double *d_in_scratch = nullptr, *d_out_scratch = nullptr;  // for host-buffer calls
  void* split = nullptr;  // split-precision state (opaque)
  su2::OpStream os;       // out-of-core operator arenas (os.on)
  su2::Profiler prof;
};

namespace su2 {
// Bytes of the split path's intermediates (T in float-float, the T' slabs) of a
// growing set of tasks, as split_prepare lays them out: the stacks are dense (all
// left blocks of a sector times all its output columns, all psi rows of a
// right sector times all its right blocks)
class SplitBytes {
 public:
  SplitBytes(const su2_env& env, int S);
  void clear();
  int64_t add(const std::vector<int64_t>& tasks);  // the bytes with these tasks too

 private:
  const su2_env& env_;
  int S_, stamp_ = 0;
  int64_t bytes_ = 0;
  std::vector<char> ham_;
  std::vector<int> f_cols_, e_rows_, d_rows_, a_seen_, d_seen_;
  std::vector<std::vector<int>> a_of_;  // the left blocks of each output sector, ascending
  std::vector<int64_t> tp_, t_;         // bytes of T' by left sector, of T by right sector
};
}  // namespace su2
