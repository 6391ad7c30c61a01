// FP64 vector kernels of the Davidson eigensolver (the diagonalisation of
// Sec. II): deterministic two-stage reductions (per-CTA partials summed in
// a fixed order), subspace combinations, preconditioner, and a one-CTA
// cyclic Jacobi eigensolver for the projected matrix (at most 32 x 32).
#include <cuda_runtime.h>

#include <cstdint>

namespace su2 {
namespace {

constexpr int kMaxSub = 32;
constexpr int kRedThreads = 256;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// partial[i * gridDim.x + blockIdx.x] = sum over this CTA's slice of V_i . w,
// eight vectors at a time (w is read again from L1 for the next eight): all 32
// accumulators at once took 255 registers, one CTA per SM and 50 us for four
// vectors that L2 holds
constexpr int kDotGroup = 8;
__device__ __forceinline__ void dot_slices(const double* V, int64_t ldv, int nvec, const double* w, int64_t n,
                                           double (*red)[kMaxSub], double* __restrict__ partial) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t stride = int64_t(gridDim.x) * blockDim.x;
  for (int v0 = 0; v0 < nvec; v0 += kDotGroup) {
    double acc[kDotGroup];
#pragma unroll
    for (int i = 0; i < kDotGroup; ++i) acc[i] = 0.0;
#pragma unroll 2
    for (int64_t x = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; x < n; x += stride) {
      const double wx = w[x];
#pragma unroll
      for (int i = 0; i < kDotGroup; ++i)
        if (v0 + i < nvec) acc[i] = fma(V[(v0 + i) * ldv + x], wx, acc[i]);
    }
#pragma unroll
    for (int i = 0; i < kDotGroup; ++i) {
      if (v0 + i >= nvec) break;
      const double s = warp_sum(acc[i]);
      if (lane == 0) red[wid][v0 + i] = s;
    }
  }
  __syncthreads();
  if (threadIdx.x < nvec) {
    double s = 0.0;
    for (int q = 0; q < kRedThreads / 32; ++q) s += red[q][threadIdx.x];
    partial[int64_t(threadIdx.x) * gridDim.x + blockIdx.x] = s;
  }
}

// sum of ng partials of one vector by a whole warp (lane-strided, then a fixed shuffle tree); valid in lane 0
__device__ __forceinline__ double sum_partials(const double* __restrict__ p, int ng) {
  double s = 0.0;
#pragma unroll 8
  for (int g = threadIdx.x & 31; g < ng; g += 32) s += p[g];
  return warp_sum(s);
}

__global__ void __launch_bounds__(kRedThreads) multidot_kernel(const double* __restrict__ V, int64_t ldv, int nvec,
                                                               const double* __restrict__ w, int64_t n,
                                                               double* __restrict__ partial, const int* __restrict__ dn) {
  if (dn) nvec = *dn + nvec;
  __shared__ double red[kRedThreads / 32][kMaxSub];
  dot_slices(V, ldv, nvec, w, n, red, partial);
}

// out[i] = sum_g partial[i * ng + g], one warp per vector (one thread walking
// the 1216 partials of a vector took 80 us, six times per iteration)
__global__ void __launch_bounds__(1024) reduce_partials_kernel(const double* __restrict__ partial, int ng, int nvec,
                                                               double* __restrict__ out, const int* __restrict__ dn) {
  if (dn) nvec = *dn + nvec;
  const int i = threadIdx.x >> 5;
  if (i >= nvec) return;
  const double s = sum_partials(partial + int64_t(i) * ng, ng);
  if ((threadIdx.x & 31) == 0) out[i] = s;
}

// out = sum_i y[i] V_i    (and optionally out2 = sum_i y[i] W_i)
__global__ void combine_kernel(const double* __restrict__ V, const double* __restrict__ W, int64_t ldv, int nvec,
                               const double* __restrict__ y, int64_t n, double* __restrict__ out,
                               double* __restrict__ out2, const int* __restrict__ dn) {
  if (dn) nvec = *dn + nvec;
  __shared__ double sy[kMaxSub];
  if (threadIdx.x < nvec) sy[threadIdx.x] = y[threadIdx.x];
  __syncthreads();
  const int64_t stride = int64_t(gridDim.x) * blockDim.x;
  for (int64_t x = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; x < n; x += stride) {
    double a = 0.0, b = 0.0;
    for (int i = 0; i < nvec; ++i) {
      a = fma(sy[i], V[i * ldv + x], a);
      if (W) b = fma(sy[i], W[i * ldv + x], b);
    }
    out[x] = a;
    if (W) out2[x] = b;
  }
}

// t -= sum_i h[i] V_i, then the partial sums of V_i . t (norm = 0) or of t . t
// (norm = 1) of the new t (a thread reads back the elements it wrote; the
// second read of V hits L2)
__global__ void __launch_bounds__(kRedThreads) ortho_kernel(const double* __restrict__ V, int64_t ldv, int nvec,
                                                            const double* __restrict__ h, int64_t n, int norm,
                                                            double* t, double* __restrict__ partial,
                                                            const int* __restrict__ dn) {
  if (dn) nvec = *dn + nvec;
  __shared__ double sh[kMaxSub], red[kRedThreads / 32][kMaxSub];
  if (threadIdx.x < nvec) sh[threadIdx.x] = h[threadIdx.x];
  __syncthreads();
  const int64_t stride = int64_t(gridDim.x) * blockDim.x;
#pragma unroll 2
  for (int64_t x = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; x < n; x += stride) {
    double a = t[x];
#pragma unroll 8
    for (int i = 0; i < nvec; ++i) a = fma(-sh[i], V[i * ldv + x], a);
    t[x] = a;
  }
  if (norm) dot_slices(t, 0, 1, t, n, red, partial);
  else dot_slices(V, ldv, nvec, t, n, red, partial);
}

// Ritz pair, residual and correction in one pass: x = V y, r = AV y - theta x,
// t = r / (diag - theta) with |diag - theta| clamped to >= 1e-12 (sign kept),
// and the partial sums of r . r
__global__ void __launch_bounds__(kRedThreads) ritz_kernel(const double* __restrict__ V, const double* __restrict__ W,
                                                           int64_t ldv, int nvec, const double* __restrict__ y,
                                                           const double* __restrict__ theta,
                                                           const double* __restrict__ diag, int64_t n,
                                                           double* __restrict__ xout, double* __restrict__ t,
                                                           double* __restrict__ partial, const int* __restrict__ dn) {
  if (dn) nvec = *dn + nvec;
  __shared__ double sy[kMaxSub], red[kRedThreads / 32];
  if (threadIdx.x < nvec) sy[threadIdx.x] = y[threadIdx.x];
  __syncthreads();
  const double th = *theta;
  double acc = 0.0;
  const int64_t stride = int64_t(gridDim.x) * blockDim.x;
  for (int64_t x = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; x < n; x += stride) {
    double a = 0.0, b = 0.0;
#pragma unroll 8
    for (int i = 0; i < nvec; ++i) {
      a = fma(sy[i], V[i * ldv + x], a);
      b = fma(sy[i], W[i * ldv + x], b);
    }
    const double r = fma(-th, a, b);
    double d = diag[x] - th;
    if (fabs(d) < 1e-12) d = d >= 0.0 ? 1e-12 : -1e-12;
    xout[x] = a;
    t[x] = r / d;
    acc = fma(r, r, acc);
  }
  acc = warp_sum(acc);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int q = 0; q < kRedThreads / 32; ++q) s += red[q];
    partial[blockIdx.x] = s;
  }
}

// r = ax - theta x
__global__ void residual_kernel(const double* __restrict__ x, const double* __restrict__ ax,
                                const double* __restrict__ theta, int64_t n, double* __restrict__ r) {
  const double th = *theta;
  const int64_t stride = int64_t(gridDim.x) * blockDim.x;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += stride) r[i] = fma(-th, x[i], ax[i]);
}

// y = x * s[0]^(-1/2) when s holds a squared norm
__global__ void scale_kernel(double* __restrict__ y, const double* __restrict__ x, const double* __restrict__ nrm2,
                             int64_t n) {
  const double s = 1.0 / sqrt(*nrm2);
  const int64_t stride = int64_t(gridDim.x) * blockDim.x;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += stride) y[i] = x[i] * s;
}

// Rayleigh-Ritz of the subspace: the new column of the projected matrix H
// (leading dim ld) from the partial sums of V_i . A V_(n-1), then cyclic Jacobi
// on its symmetrised n x n part; ascending eigenvalues w and eigenvectors Y
// (column j, ld rows).  One CTA; the n / 2 rotations of a round (round-robin
// order) act on disjoint rows and columns and run side by side, one warp each.
// A rotation's tangent is taken in FP32 (from entries scaled to their common
// exponent) and c = 1 / sqrt(1 + t^2), s = t c in FP64: orthogonal to FP64
// accuracy, while the annihilated entry is left at 1e-7 of its size for the
// next sweep.  One rotation after another, each with FP64 divisions and square
// roots by one thread, took about 1.7 us a rotation, 2 to 3 ms at n = 24.
__global__ void __launch_bounds__(1024) rayleigh_kernel(double* __restrict__ H, int ld, int n,
                                                        const double* __restrict__ partial, int ng,
                                                        double* __restrict__ w, double* __restrict__ Y,
                                                        int* __restrict__ status, const int* __restrict__ dn) {
  if (dn) n = *dn + n;
  __shared__ double A[kMaxSub][kMaxSub + 1], V[kMaxSub][kMaxSub + 1];
  __shared__ double soff[32], stot[32];
  __shared__ int done;
  const int t = threadIdx.x & 31, k = threadIdx.x >> 5;
  if (k < n) {
    const double h = sum_partials(partial + int64_t(k) * ng, ng);
    if (t == 0) {
      H[k + (n - 1) * ld] = h;
      H[(n - 1) + k * ld] = h;
    }
  }
  __syncthreads();
  if (k < n && t < n) {
    A[k][t] = 0.5 * (H[k + t * ld] + H[t + k * ld]);
    V[k][t] = (k == t) ? 1.0 : 0.0;
  }
  if (threadIdx.x == 0) done = 0;
  __syncthreads();
  const int m = n + (n & 1);  // (an odd n plays against a dummy)
  for (int sweep = 0; sweep < 60; ++sweep) {
    const double v = (k < n && t < n) ? A[k][t] : 0.0;
    const double o = warp_sum(k == t ? 0.0 : v * v), d = warp_sum(v * v);
    if (t == 0) {
      soff[k] = o;
      stot[k] = d;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
      const double off = warp_sum(soff[t]), tot = warp_sum(stot[t]);
      if (t == 0) done = (off <= 1e-30 * tot) || tot == 0.0;
    }
    __syncthreads();
    if (done) break;
    for (int r = 0; r < m - 1; ++r) {
      int p = 0, q = 0;
      double c = 1.0, s = 0.0;
      if (k < m / 2) {
        p = k == 0 ? m - 1 : (r + k) % (m - 1);
        q = k == 0 ? r : (r + m - 1 - k) % (m - 1);
        if (p > q) {
          const int x = p;
          p = q;
          q = x;
        }
        if (q < n) {
          const double apq = A[p][q], df = A[q][q] - A[p][p];
          // common scale: the larger of the two gets exponent 0
          const int be = max((__double2hiint(apq) >> 20) & 0x7FF, (__double2hiint(df) >> 20) & 0x7FF);
          const double sc = __longlong_as_double((long long)min(2046, max(1, 2046 - be)) << 52);
          const float fa = (float)(apq * sc), fd = (float)(df * sc);
          if (fa != 0.f) {
            const float tau = fd / (2.f * fa);
            float tt = fabsf(tau) > 1e9f ? 0.5f / fabsf(tau) : 1.f / (fabsf(tau) + sqrtf(1.f + tau * tau));
            if (tau < 0.f) tt = -tt;
            const double td = tt, x = fma(td, td, 1.0);
            double y = rsqrtf((float)x);
            y = y * fma(-0.5 * x * y, y, 1.5);
            y = y * fma(-0.5 * x * y, y, 1.5);
            c = y;
            s = td * y;
          }
        }
      }
      __syncthreads();
      if (s != 0.0 && t < n) {  // columns p, q
        const double akp = A[t][p], akq = A[t][q];
        A[t][p] = c * akp - s * akq;
        A[t][q] = s * akp + c * akq;
        const double vkp = V[t][p], vkq = V[t][q];
        V[t][p] = c * vkp - s * vkq;
        V[t][q] = s * vkp + c * vkq;
      }
      __syncthreads();
      if (s != 0.0 && t < n) {  // rows p, q
        const double apk = A[p][t], aqk = A[q][t];
        A[p][t] = c * apk - s * aqk;
        A[q][t] = s * apk + c * aqk;
      }
      __syncthreads();
    }
  }
  if (k < n) {  // eigenpair k to its place in ascending order (ties: by index)
    int rank = 0;
    const double e = A[k][k];
    for (int j = 0; j < n; ++j) rank += A[j][j] < e || (A[j][j] == e && j < k);
    if (t == 0) w[rank] = e;
    if (t < n) Y[t + rank * ld] = V[t][k];
  }
  if (threadIdx.x == 0 && !done) *status = 4;
}

// partial max |x| and its index per CTA
__global__ void absmax_kernel(const double* __restrict__ x, int64_t n, double* __restrict__ pv,
                              int64_t* __restrict__ pi) {
  __shared__ double sv[256];
  __shared__ int64_t si[256];
  double best = -1.0;
  int64_t bi = 0;
  const int64_t stride = int64_t(gridDim.x) * blockDim.x;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += stride) {
    const double a = fabs(x[i]);
    if (a > best) { best = a; bi = i; }
  }
  sv[threadIdx.x] = best;
  si[threadIdx.x] = bi;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
      const double a = sv[threadIdx.x + o];
      const int64_t ai = si[threadIdx.x + o];
      if (a > sv[threadIdx.x] || (a == sv[threadIdx.x] && ai < si[threadIdx.x])) {
        sv[threadIdx.x] = a;
        si[threadIdx.x] = ai;
      }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    pv[blockIdx.x] = sv[0];
    pi[blockIdx.x] = si[0];
  }
}

__global__ void diag_set_kernel(double* __restrict__ H, int ld, int n, const double* __restrict__ w) {
  for (int idx = threadIdx.x; idx < ld * ld; idx += blockDim.x) {
    const int i = idx % ld, j = idx / ld;
    H[idx] = (i == j && i < n) ? w[i] : 0.0;
  }
}

// ---- device-side subspace bookkeeping (graph-capturable Davidson iteration)
// dst = V[nsub-1] (dir 0) or V[nsub-1] = src (dir 1)
__global__ void newest_copy_kernel(double* __restrict__ V, int64_t n, const int* __restrict__ dn,
                                   double* __restrict__ w, int dir) {
  const int64_t base = int64_t(*dn - 1) * n;
  const int64_t stride = int64_t(gridDim.x) * blockDim.x;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += stride) {
    if (dir == 0) w[i] = V[base + i];
    else V[base + i] = w[i];
  }
}

// restart when the subspace is full: V[q] <- V Y[:, q], AV[q] <- AV Y[:, q]
// for q < keep (into tmp, then back), H <- diag(w[:keep]); sets *dn = keep
__global__ void restart_combine_kernel(const double* __restrict__ V, const double* __restrict__ AV, int64_t n,
                                       const double* __restrict__ Y, int ld, int keep, int max_sub,
                                       const int* __restrict__ dn, double* __restrict__ tmp) {
  if (*dn < max_sub) return;
  const int nv = *dn;
  const int64_t stride = int64_t(gridDim.x) * blockDim.x;
  for (int64_t x = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; x < n; x += stride)
    for (int q = 0; q < keep; ++q) {
      double a = 0.0, b = 0.0;
      for (int i = 0; i < nv; ++i) {
        a = fma(Y[i + q * ld], V[int64_t(i) * n + x], a);
        b = fma(Y[i + q * ld], AV[int64_t(i) * n + x], b);
      }
      tmp[int64_t(2 * q) * n + x] = a;
      tmp[int64_t(2 * q + 1) * n + x] = b;
    }
}
__global__ void restart_copy_kernel(double* __restrict__ V, double* __restrict__ AV, int64_t n, int keep, int max_sub,
                                    const int* __restrict__ dn, const double* __restrict__ tmp) {
  if (*dn < max_sub) return;
  const int64_t stride = int64_t(gridDim.x) * blockDim.x;
  for (int64_t x = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; x < n; x += stride)
    for (int q = 0; q < keep; ++q) {
      V[int64_t(q) * n + x] = tmp[int64_t(2 * q) * n + x];
      AV[int64_t(q) * n + x] = tmp[int64_t(2 * q + 1) * n + x];
    }
}
__global__ void restart_finish_kernel(double* __restrict__ H, int ld, const double* __restrict__ w, int keep,
                                      int max_sub, int* __restrict__ dn) {
  if (*dn < max_sub) return;
  __syncthreads();
  for (int idx = threadIdx.x; idx < ld * ld; idx += blockDim.x) {
    const int i = idx % ld, j = idx / ld;
    H[idx] = (i == j && i < keep) ? w[i] : 0.0;
  }
  __syncthreads();
  if (threadIdx.x == 0) *dn = keep;
}
// V[nsub] = t / ||t|| when ||t||^2 > tiny (else the subspace is left as is)
__global__ void append_kernel(double* __restrict__ V, int64_t n, const int* __restrict__ dn,
                              const double* __restrict__ t, const double* __restrict__ nrm2) {
  if (!(*nrm2 > 1e-28)) return;
  const double s = 1.0 / sqrt(*nrm2);
  const int64_t base = int64_t(*dn) * n;
  const int64_t stride = int64_t(gridDim.x) * blockDim.x;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += stride) V[base + i] = t[i] * s;
}
__global__ void append_count_kernel(int* __restrict__ dn, const double* __restrict__ nrm2) {
  if (threadIdx.x == 0 && *nrm2 > 1e-28) *dn += 1;
}

}  // namespace

// CTAs of a vector kernel: about four elements per thread while that fills the
// chip, at most four CTAs per SM (fewer partial sums to add up afterwards)
int dav_grid(int64_t n) {
  const int64_t g = (n + 1023) / 1024, most = 152 * 4, least = (n + 255) / 256;
  return int(g >= 152 ? (g > most ? most : g) : least < 1 ? 1 : (least > 152 ? 152 : least));
}

// partial sums of V_i . w; out (if given) gets the sums
void dav_multidot(cudaStream_t s, const double* V, int64_t ldv, int nvec, const double* w, int64_t n,
                  double* partial, double* out, const int* dn) {
  const int g = dav_grid(n);
  multidot_kernel<<<g, kRedThreads, 0, s>>>(V, ldv, nvec, w, n, partial, dn);
  if (out) reduce_partials_kernel<<<1, 1024, 0, s>>>(partial, g, nvec, out, dn);
}
// t -= V h, then out = V^T t, or t . t with norm
void dav_ortho(cudaStream_t s, const double* V, int64_t ldv, int nvec, const double* h, int64_t n, bool norm, double* t,
               double* partial, double* out, const int* dn) {
  const int g = dav_grid(n);
  ortho_kernel<<<g, kRedThreads, 0, s>>>(V, ldv, nvec, h, n, norm ? 1 : 0, t, partial, dn);
  reduce_partials_kernel<<<1, 1024, 0, s>>>(partial, g, norm ? 1 : nvec, out, norm ? nullptr : dn);
}
// x = V y, t = (AV y - theta x) / (diag - theta), out = || AV y - theta x ||^2
void dav_ritz(cudaStream_t s, const double* V, const double* W, int64_t ldv, int nvec, const double* y,
              const double* theta, const double* diag, int64_t n, double* x, double* t, double* partial, double* out,
              const int* dn) {
  const int g = dav_grid(n);
  ritz_kernel<<<g, kRedThreads, 0, s>>>(V, W, ldv, nvec, y, theta, diag, n, x, t, partial, dn);
  reduce_partials_kernel<<<1, 1024, 0, s>>>(partial, g, 1, out, nullptr);
}
// Rayleigh-Ritz from the partial sums of the last dav_multidot
void dav_rayleigh(cudaStream_t s, double* H, int ld, int n, const double* partial, int64_t nvecs, double* w, double* Y,
                  int* status, const int* dn) {
  rayleigh_kernel<<<1, 1024, 0, s>>>(H, ld, n, partial, dav_grid(nvecs), w, Y, status, dn);
}
void dav_combine(cudaStream_t s, const double* V, const double* W, int64_t ldv, int nvec, const double* y, int64_t n,
                 double* out, double* out2, const int* dn) {
  combine_kernel<<<dav_grid(n), 256, 0, s>>>(V, W, ldv, nvec, y, n, out, out2, dn);
}
void dav_residual(cudaStream_t s, const double* x, const double* ax, const double* theta, int64_t n, double* r) {
  residual_kernel<<<dav_grid(n), 256, 0, s>>>(x, ax, theta, n, r);
}
void dav_scale(cudaStream_t s, double* y, const double* x, const double* nrm2, int64_t n) {
  scale_kernel<<<dav_grid(n), 256, 0, s>>>(y, x, nrm2, n);
}
void dav_absmax(cudaStream_t s, const double* x, int64_t n, double* pv, int64_t* pi, int* ng) {
  const int g = dav_grid(n);
  *ng = g;
  absmax_kernel<<<g, 256, 0, s>>>(x, n, pv, pi);
}
void dav_diag_set(cudaStream_t s, double* H, int ld, int n, const double* w) {
  diag_set_kernel<<<1, 256, 0, s>>>(H, ld, n, w);
}
void dav_newest(cudaStream_t s, double* V, int64_t n, const int* dn, double* w, int dir) {
  newest_copy_kernel<<<dav_grid(n), 256, 0, s>>>(V, n, dn, w, dir);
}
void dav_restart(cudaStream_t s, double* V, double* AV, int64_t n, const double* Y, int ld, double* H,
                 const double* w, int keep, int max_sub, int* dn, double* tmp) {
  restart_combine_kernel<<<dav_grid(n), 256, 0, s>>>(V, AV, n, Y, ld, keep, max_sub, dn, tmp);
  restart_copy_kernel<<<dav_grid(n), 256, 0, s>>>(V, AV, n, keep, max_sub, dn, tmp);
  restart_finish_kernel<<<1, 256, 0, s>>>(H, ld, w, keep, max_sub, dn);
}
void dav_append(cudaStream_t s, double* V, int64_t n, int* dn, const double* t, const double* nrm2) {
  append_kernel<<<dav_grid(n), 256, 0, s>>>(V, n, dn, t, nrm2);
  append_count_kernel<<<1, 32, 0, s>>>(dn, nrm2);
}

}  // namespace su2
