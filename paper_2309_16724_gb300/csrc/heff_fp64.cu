// Native-FP64 path of H.psi (Eq. 2 over the sector-task-table of Eq. 3), and
// the grouped FP64 products of the renormalisation.  Deterministic: no atomics.
//
// H.psi: GB300 has two FP64 lanes per SM and clock (1.06 TFLOP/s measured), so
// everything here is bound by the number of DFMAs issued and, for small
// sectors, by how long one CTA's chain of K steps is.  Hence stacked products:
// K1 forms T = E . D^T of one input block with all its right blocks side by
// side; K2 is output stationary over the output blocks of one left sector side
// by side, with the left blocks of that sector along K and the tasks that
// share a left and an output block summed while the tile is filled (1.7 to 3
// times fewer DFMAs than one product per task, Sec. III.A's stripe).  Rows past
// a block are skipped warp by warp and columns sixteen at a time; the K of a
// tile is split over several CTAs when the tiles alone leave the chip idle.
#include "su2_device.h"

namespace su2 {
namespace {

constexpr int TK = 16;
constexpr int NT = 256;

// acc(row, col) += sum_kk A(kk, row) B(kk, col), thread (tx, ty) owning rows
// ty + 16 i, i < NI, and columns tx + 16 j, j < NJ.  NI is uniform in a warp
// (two rows of ty) and NJ in the CTA, and both are template parameters: a
// DFMA that is predicated off for a whole warp still takes its slot in the
// FP64 pipe (measured: 91 % busy at 54 % useful lanes)
template <int NI, int NJ>
__device__ __forceinline__ void fma_step(double (&acc)[4][4], const double (*sA)[kTile], const double (*sB)[kTile],
                                         int tx, int ty, int kend) {
#pragma unroll 4
  for (int kk = 0; kk < kend; ++kk) {
    double b[NJ];
#pragma unroll
    for (int j = 0; j < NJ; ++j) b[j] = sB[kk][tx + 16 * j];
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      const double a = sA[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < NJ; ++j) acc[i][j] = fma(a, b[j], acc[i][j]);
    }
  }
}
template <int NJ>
__device__ __forceinline__ void fma_rows(double (&acc)[4][4], const double (*sA)[kTile], const double (*sB)[kTile],
                                         int tx, int ty, int kend, int ni) {
  if (ni == 4) fma_step<4, NJ>(acc, sA, sB, tx, ty, kend);
  else if (ni == 3) fma_step<3, NJ>(acc, sA, sB, tx, ty, kend);
  else if (ni == 2) fma_step<2, NJ>(acc, sA, sB, tx, ty, kend);
  else if (ni == 1) fma_step<1, NJ>(acc, sA, sB, tx, ty, kend);
}
__device__ __forceinline__ void fma_tile(double (&acc)[4][4], const double (*sA)[kTile], const double (*sB)[kTile],
                                         int tx, int ty, int kend, int ni, int nj) {
  if (nj == 4) fma_rows<4>(acc, sA, sB, tx, ty, kend, ni);
  else if (nj == 3) fma_rows<3>(acc, sA, sB, tx, ty, kend, ni);
  else if (nj == 2) fma_rows<2>(acc, sA, sB, tx, ty, kend, ni);
  else fma_rows<1>(acc, sA, sB, tx, ty, kend, ni);
}
// row slots of this warp below `rows` (its lower row is ty & ~1)
__device__ __forceinline__ int row_slots(int ty, int rows) { return max(0, min(4, (rows - (ty & ~1) + 15) >> 4)); }

// acc += alpha * A(r0:r0+64, 0:K) . B(0:K, c0:c0+64); A column-major (lda),
// B(kk, c) = BT ? B[c + kk*ldb] : B[kk + c*ldb].  Out-of-range entries are 0.
template <bool BT>
__device__ __forceinline__ void tile_gemm(double (&acc)[4][4], const double* __restrict__ A, int lda,
                                          const double* __restrict__ B, int ldb, int M, int N, int K, int r0, int c0,
                                          double alpha, double (*sA)[kTile], double (*sB)[kTile]) {
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int ni = row_slots(ty, M - r0), nj = (min(kTile, N - c0) + 15) / 16;
  for (int k0 = 0; k0 < K; k0 += TK) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int idx = tid + NT * i;
      const int r = idx & 63, kk = idx >> 6;
      const int gr = r0 + r, gk = k0 + kk;
      sA[kk][r] = (gr < M && gk < K) ? alpha * A[gr + int64_t(gk) * lda] : 0.0;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int idx = tid + NT * i;
      int kk, c;
      if (BT) {
        c = idx & 63;
        kk = idx >> 6;
      } else {
        kk = idx & 15;
        c = idx >> 4;
      }
      const int gc = c0 + c, gk = k0 + kk;
      double v = 0.0;
      if (gc < N && gk < K) v = BT ? B[gc + int64_t(gk) * ldb] : B[gk + int64_t(gc) * ldb];
      sB[kk][c] = v;
    }
    __syncthreads();
    fma_tile(acc, sA, sB, tx, ty, min(TK, K - k0), ni, nj);
    __syncthreads();
  }
}

__global__ void __launch_bounds__(NT) k1_fp64(const K1Job* __restrict__ jobs, const double* __restrict__ psi,
                                              const double* __restrict__ R, double* __restrict__ T) {
  __shared__ double sA[TK][kTile], sB[TK][kTile];
  const K1Job j = jobs[blockIdx.x];
  double acc[4][4] = {};
  const int r0 = j.tr * kTile, c0 = j.tc * kTile;
  tile_gemm<true>(acc, psi + j.e_off, j.k1, R + j.d_off, j.n, j.k1, j.n, j.k2, r0, c0, 1.0, sA, sB);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int jj = 0; jj < 4; ++jj) {
      const int r = r0 + ty + 16 * i, c = c0 + tx + 16 * jj;
      if (r < j.k1 && c < j.n) T[j.t_off + r + int64_t(c) * j.k1] = acc[i][jj];
    }
}

__global__ void __launch_bounds__(NT) k2_fp64(const K2Job* __restrict__ jobs, const K2Task* __restrict__ tasks,
                                              const double* __restrict__ L, const double* __restrict__ T,
                                              double* __restrict__ F, double* __restrict__ part) {
  __shared__ double sA[TK][kTile], sB[TK][kTile];
  const K2Job j = jobs[blockIdx.x];
  const int r0 = j.tr * kTile, c0 = j.tc * kTile;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double acc[4][4] = {};
  for (int t = j.t0; t < j.t1; ++t) {
    const K2Task task = tasks[t];
    tile_gemm<false>(acc, L + task.a_off, j.m, T + task.b_off, task.k1, j.m, j.n, task.k1, r0, c0, task.v, sA, sB);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int jj = 0; jj < 4; ++jj) {
      const int r = r0 + ty + 16 * i, c = c0 + tx + 16 * jj;
      if (r >= j.m || c >= j.n) continue;
      if (j.part >= 0) part[j.part + (c - c0) * min(kTile, j.m - r0) + (r - r0)] = acc[i][jj];
      else F[j.f_off + r + int64_t(c) * j.m] += acc[i][jj];
    }
}

// ------------------------------------------------------------------ stacked H.psi
// the entry of [lo, hi) that holds column c (col0 ascending, col0[lo] <= c)
__device__ __forceinline__ int find_ent(const P64Ent* __restrict__ ents, int lo, int hi, int c) {
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (ents[mid].col0 <= c) lo = mid;
    else hi = mid;
  }
  return lo;
}

__global__ void __launch_bounds__(NT, 2) k1_stack(const P64K1* __restrict__ jobs, const P64In* __restrict__ ins,
                                                  const P64Ent* __restrict__ ents, const double* __restrict__ psi,
                                                  const double* __restrict__ R, double* __restrict__ T) {
  __shared__ double sA[TK][kTile], sB[TK][kTile];
  const P64K1 j = jobs[blockIdx.x];
  const P64In p = ins[j.in];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int r0 = j.tr * kTile, c0 = j.tc * kTile, last = min(p.ent1, j.ent + kTile);
  // fill: row (A) and column (B) tid & 63, K tid >> 6 + 4 i
  const int gr = r0 + (tid & 63), gc = c0 + (tid & 63), kq = tid >> 6;
  const double* ap = gr < p.k1 ? psi + p.e_off + gr : nullptr;
  const double* bp = nullptr;
  int ldb = 0;
  if (gc < p.ncol) {
    const P64Ent e = ents[find_ent(ents, j.ent, last, gc)];
    bp = R + e.d_off + (gc - e.col0);
    ldb = e.n;
  }
  double ra[4], rb[4];
  auto load = [&](int k0) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int k = k0 + kq + 4 * i;
      ra[i] = ap && k < p.k2 ? ap[int64_t(k) * p.k1] : 0.0;
      rb[i] = bp && k < p.k2 ? bp[int64_t(k) * ldb] : 0.0;
    }
  };
  double acc[4][4] = {};
  bool on[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) on[i] = r0 + ty + 16 * i < p.k1;
  const int ni = row_slots(ty, p.k1 - r0), nj = (min(kTile, p.ncol - c0) + 15) / 16;
  load(0);
  for (int k0 = 0; k0 < p.k2; k0 += TK) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      sA[kq + 4 * i][tid & 63] = ra[i];
      sB[kq + 4 * i][tid & 63] = rb[i];
    }
    __syncthreads();
    if (k0 + TK < p.k2) load(k0 + TK);
    fma_tile(acc, sA, sB, tx, ty, min(TK, p.k2 - k0), ni, nj);
    __syncthreads();
  }
#pragma unroll
  for (int jj = 0; jj < 4; ++jj) {
    const int c = c0 + tx + 16 * jj;
    if (c >= p.ncol) break;
    const P64Ent e = ents[find_ent(ents, j.ent, last, c)];
    double* t = T + e.t_off + int64_t(c - e.col0) * p.k1;
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (on[i]) t[r0 + ty + 16 * i] = acc[i][jj];
  }
}

struct KMeta { int64_t a; int32_t w, k; };  // one K of a step: column of the A stack, left block (-1: past the end), K within it

__global__ void __launch_bounds__(NT, 2) k2_stack(const P64K2* __restrict__ jobs, const P64Stack* __restrict__ stacks,
                                                  const P64Left* __restrict__ lefts, const int32_t* __restrict__ steps,
                                                  const int32_t* __restrict__ tab, const P64Task* __restrict__ tasks,
                                                  const P64Col* __restrict__ cols, const double* __restrict__ L,
                                                  const double* __restrict__ psi, const double* __restrict__ T,
                                                  double* __restrict__ F, double* __restrict__ part) {
  __shared__ double sA[TK][kTile], sB[TK][kTile];
  __shared__ KMeta meta[2][TK];
  const P64K2 j = jobs[blockIdx.x];
  const P64Stack s = stacks[j.st];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int r0 = j.tr * kTile, c0 = j.tc * kTile;
  const P64Left* lf = lefts + s.left0;
  auto fill_meta = [&](int st) {  // threads 0 .. 15
    if (tid < TK) {
      const int kg = st * TK + tid;
      KMeta m{0, -1, 0};
      if (kg < s.K) {
        int w = steps[s.step0 + st];
        while (lf[w + 1].k0 <= kg) ++w;
        m.w = w;
        m.k = kg - lf[w].k0;
        m.a = lf[w].a_off < 0 ? int64_t(-1 - m.k) : lf[w].a_off + int64_t(m.k) * s.m;
      }
      meta[st & 1][tid] = m;
    }
  };
  // fill: A row tid & 63, K tid >> 6 + 4 i; B K tid & 15 (neighbouring lanes
  // read neighbouring rows of T), columns tid >> 4 + 16 i
  const int gr = r0 + (tid & 63), kq = tid >> 6, kb = tid & 15;
  const int32_t* tb[4];
  int cc[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int c = c0 + (tid >> 4) + 16 * i;
    tb[i] = nullptr;
    cc[i] = 0;
    if (c < s.N) {
      const P64Col cm = cols[s.col0 + c];
      tb[i] = tab + s.tab_off + cm.f;
      cc[i] = cm.c;
    }
  }
  double ra[4], rb[4];
  auto load = [&](int st) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const KMeta m = meta[st & 1][kq + 4 * i];
      ra[i] = 0.0;
      if (m.w >= 0 && gr < s.m) ra[i] = m.a >= 0 ? L[m.a + gr] : (gr == int(-1 - m.a) ? 1.0 : 0.0);
    }
    const KMeta m = meta[st & 1][kb];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      rb[i] = 0.0;
      if (m.w >= 0 && tb[i]) {
        const int t1 = tb[i][int64_t(m.w) * s.nf + 1];
        for (int t = tb[i][int64_t(m.w) * s.nf]; t < t1; ++t) {
          const P64Task tk = tasks[t];
          rb[i] = fma(tk.v, (tk.psi ? psi : T)[tk.off + m.k + int64_t(cc[i]) * tk.ld], rb[i]);
        }
      }
    }
  };
  double acc[4][4] = {};
  bool on[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) on[i] = r0 + ty + 16 * i < s.m;
  const int ni = row_slots(ty, s.m - r0), nj = (min(kTile, s.N - c0) + 15) / 16;
  fill_meta(j.s0);
  fill_meta(j.s0 + 1);
  __syncthreads();
  load(j.s0);
  for (int st = j.s0; st < j.s1; ++st) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      sA[kq + 4 * i][tid & 63] = ra[i];
      sB[kb][(tid >> 4) + 16 * i] = rb[i];
    }
    __syncthreads();  // (every thread has used meta[st & 1])
    fill_meta(st + 2);
    if (st + 1 < j.s1) load(st + 1);
    fma_tile(acc, sA, sB, tx, ty, min(TK, s.K - st * TK), ni, nj);
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int jj = 0; jj < 4; ++jj) {
      const int r = ty + 16 * i, c = tx + 16 * jj;
      if (!on[i] || c0 + c >= s.N) continue;
      if (j.part >= 0) part[j.part + c * min(kTile, s.m - r0) + r] = acc[i][jj];
      else F[s.f_off + r0 + r + int64_t(c0 + c) * s.m] += acc[i][jj];
    }
}

// F += the partial tiles of the tiles whose K was split, in K order
__global__ void __launch_bounds__(NT) part_sum(const P64Tile* __restrict__ tiles, const double* __restrict__ part,
                                               double* __restrict__ F) {
  const P64Tile t = tiles[blockIdx.x];
  const int r = threadIdx.x & 63;
  if (r >= t.rows) return;
  for (int c = threadIdx.x >> 6; c < t.cols; c += NT / 64) {
    double x = 0.0;
#pragma unroll 4
    for (int i = 0; i < t.npart; ++i) x += part[t.part0 + int64_t(i) * t.rows * t.cols + c * t.rows + r];
    F[t.f_off + r + int64_t(c) * t.ld] += x;
  }
}

// diag(H_eff) of one 64 x 64 tile of a psi block: sum_t v_t a_t(r) d_t(c), an
// outer-product sum with the diagonal tasks along K.  (One thread per element
// walking the tasks read both diagonals from L2 for every element: 177 ms at
// L = 32, D = 2048, as long as an H.psi; tiled, the diagonals are read once per
// tile and the sum runs at the DFMA rate.)
__global__ void __launch_bounds__(NT, 2) diag_kernel(const DiagJob* __restrict__ jobs, const DiagTask* __restrict__ tasks,
                                                     const double* __restrict__ L, const double* __restrict__ R,
                                                     double* __restrict__ d) {
  __shared__ double sA[TK][kTile], sB[TK][kTile];
  const DiagJob j = jobs[blockIdx.x];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4, kq = tid >> 6;
  const int r0 = j.tr * kTile, c0 = j.tc * kTile, r = r0 + (tid & 63), c = c0 + (tid & 63);
  double ra[4], rb[4];
  auto load = [&](int t0) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int t = t0 + kq + 4 * i;
      ra[i] = rb[i] = 0.0;
      if (t < j.t1) {
        const DiagTask tk = tasks[t];
        if (r < j.m) ra[i] = tk.v * (tk.a_off < 0 ? 1.0 : L[tk.a_off + r + int64_t(r) * tk.lda]);
        if (c < j.n) rb[i] = tk.d_off < 0 ? 1.0 : R[tk.d_off + c + int64_t(c) * tk.ldd];
      }
    }
  };
  double acc[4][4] = {};
  bool on[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) on[i] = r0 + ty + 16 * i < j.m;
  const int ni = row_slots(ty, j.m - r0), nj = (min(kTile, j.n - c0) + 15) / 16;
  load(j.t0);
  for (int t = j.t0; t < j.t1; t += TK) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      sA[kq + 4 * i][tid & 63] = ra[i];
      sB[kq + 4 * i][tid & 63] = rb[i];
    }
    __syncthreads();
    if (t + TK < j.t1) load(t + TK);
    fma_tile(acc, sA, sB, tx, ty, min(TK, j.t1 - t), ni, nj);
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int jj = 0; jj < 4; ++jj) {
      const int cc = c0 + tx + 16 * jj;
      if (on[i] && cc < j.n) d[j.f_off + r0 + ty + 16 * i + int64_t(cc) * j.m] = acc[i][jj];
    }
}

}  // namespace

void launch_heff_fp64(cudaStream_t s, const double* L, const double* R, const double* psi, double* F, double* T,
                      const K1Job* k1, const K2Job* k2, const K2Task* tasks, const P64Tile* split, double* part,
                      const Chunk& c) {
  const int64_t n1 = c.k1_end - c.k1_begin, n2 = c.k2_end - c.k2_begin, n3 = c.sp_end - c.sp_begin;
  if (n1 > 0) k1_fp64<<<unsigned(n1), NT, 0, s>>>(k1 + c.k1_begin, psi, R, T);
  if (n2 > 0) k2_fp64<<<unsigned(n2), NT, 0, s>>>(k2 + c.k2_begin, tasks, L, T, F, part);
  if (n3 > 0) part_sum<<<unsigned(n3), NT, 0, s>>>(split + c.sp_begin, part, F);
}

void launch_stack_fp64(cudaStream_t s, const Plan64& p, const Chunk64& c, const double* L, const double* R,
                       const double* psi, double* F, double* T, Profiler* prof) {
  const int64_t n1 = c.k1_end - c.k1_begin, n2 = c.k2_end - c.k2_begin, n3 = c.sp_end - c.sp_begin;
  prof->count(int(n1 > 0) + int(n2 > 0) + int(n3 > 0));
  if (n1 > 0) {
    const int slot = prof->begin(s, 0, c.k1_flops);
    k1_stack<<<unsigned(n1), NT, 0, s>>>(p.d_k1 + c.k1_begin, p.d_in, p.d_ent, psi, R, T);
    prof->end(s, slot);
  }
  if (n2 > 0) {
    const int slot = prof->begin(s, 1, c.k2_flops);
    k2_stack<<<unsigned(n2), NT, 0, s>>>(p.d_k2 + c.k2_begin, p.d_stack, p.d_left, p.d_step, p.d_tab, p.d_task, p.d_col,
                                         L, psi, T, F, p.d_part);
    if (n3 > 0) part_sum<<<unsigned(n3), NT, 0, s>>>(p.d_tile + c.sp_begin, p.d_part, F);
    prof->end(s, slot);
  }
}

void launch_diag(cudaStream_t s, const double* L, const double* R, double* d, const DiagJob* jobs, int64_t njobs,
                 const DiagTask* tasks, int64_t psi_len) {
  cudaMemsetAsync(d, 0, size_t(psi_len) * sizeof(double), s);
  if (njobs > 0) diag_kernel<<<unsigned(njobs), NT, 0, s>>>(jobs, tasks, L, R, d);
}

}  // namespace su2
