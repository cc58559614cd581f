// Subspace construction on the device (Algorithm 1, "Collect gradients to build basis V_r"; Sec. 3.2
// "Guided Perturbation Sampling on Cloud"): an orthonormal basis U (rows x r, r <= 64) of the span of the r
// gradient directions collected for one tensor, given as the columns of A (rows x r fp32, row-major).
//
// Method: Cholesky QR, applied twice where one pass is not enough.  One pass forms the Gram matrix  S = A^T A  (r x r), factors it
// S = R^T R  (R upper triangular with a positive diagonal) and returns  Q = A R^-1.  In exact arithmetic that is
// the thin Q of the QR factorisation with R_kk > 0, i.e. the same basis, column for column, as a Householder QR
// with that sign convention.  In floating point the first pass loses orthogonality in proportion to the
// square of the condition number of A; the second pass, applied to the nearly orthonormal Q of the first,
// restores it to working precision.  Everything between the fp32 input and the fp32 output is carried in
// double: the Gram matrices (rows x r^2 multiply-adds, a few hundred MFLOP at most for the largest tensor of
// the paper-shaped models), the r x r factorisations and the products A R^-1.  Tall-skinny and tiny in
// arithmetic, the job is bound by reading A twice and writing U once; tensor cores would add nothing but
// rounding (their split-bf16 product is good to 2^-16, an orthogonality of 1e-6 needs more).
//
// One launch does all of it (basis_kernel): every CTA keeps its rows in shared memory as doubles through both passes, the
// partial Gram matrices meet in global memory (L2) between barriers, and each CTA factors the r x r sum for itself, since
// that is cheaper than another barrier.  Up to 4096 rows in all at rank 16, 1024 above, the grid is a single cluster of 16 or 8 CTAs, whose
// barrier is a hardware one and whose partials every CTA adds up directly; larger inputs use one CTA per SM, launched
// cooperatively, with a counter barrier and the sum of the partials spread over the grid.  The job is bound by latency (a
// 2048 x 16 input is 131 KB): the six launches, the memset and the copies of the status that it took before were 95 us a
// tensor.  The last phase also writes the tensor-core operand copies of the new basis.
// Inputs whose rows do not fit the shared memory of the whole chip (more than about 200,000 rows at rank 16, 53,000 at
// rank 64) take three kernels per pass instead:
//   gram_partial   one block per chunk of 128 rows: partial Gram matrix of the chunk, written to scratch
//   factor         one block: sums the partials in a fixed order, Cholesky factor, inverse of R, status
//   apply          one block per chunk of 128 rows: Q = A R^-1
// The summation order is fixed, so the result does not depend on the launch history.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "zgr_grid_exit.h"
#include "zgr_subspace.h"

namespace zgr {
namespace {

constexpr int kChunkRows = 128;
constexpr int kLd = 65;               // leading dimension of the shared-memory matrices (64 + 1: no bank conflicts down a column)
constexpr int kQrThreads = 256;
constexpr int kMaxR = 64;
// A pivot below this share of its column's squared norm means dependent columns: an angle of 4.5e-8 to the span of the earlier
// ones.  The fp32 rounding of an exact linear combination leaves up to about 3e-8 (8e-16 here), the sums in double below 5e-16 when
// exact; directions at 5e-8 and more give a basis that is right to 3e-8 and are accepted.
constexpr double kPivotFloor = 2e-15;

// One pass is enough when it leaves the columns orthonormal far below the fp32 rounding of the result.  Errors of the Gram matrix, |dS_kl| <=
// g |a_k| |a_l| with g about 1e-15 (sums in double over at most some hundred rows, then over the CTAs), come out of the first pass as
// R^-T dS R^-1, at most g (sum_k |a_k| |R^-1_kj|)^2 <= g r m_j with m_j = sum_k |a_k|^2 (R^-1)_kj^2, which the factorisation has at
// hand.  r m_j <= 1e5 (condition numbers up to about 100 after scaling the columns to one length) keeps that near 1e-10; one fp32
// rounding is 6e-8 of an entry.  2048 x 16, mixed Gaussian directions: r m_j is about 30.
constexpr double kOnePass = 1e5;

// Partial Gram matrix of rows [chunk*128, +128) of X (rows x r).  X is fp32 (SRC_DOUBLE = false) or double.
template <bool SRC_DOUBLE>
__global__ void __launch_bounds__(kQrThreads) gram_partial_kernel(const void* __restrict__ Xv, int64_t rows, int r, double* __restrict__ partials) {
  extern __shared__ double dyn_smem[];
  double (*Xs)[kLd] = reinterpret_cast<double (*)[kLd]>(dyn_smem);          // [kChunkRows][kLd]
  const int64_t row0 = static_cast<int64_t>(blockIdx.x) * kChunkRows;
  const int nrows = static_cast<int>(min(static_cast<int64_t>(kChunkRows), rows - row0));
  for (int idx = threadIdx.x; idx < kChunkRows * r; idx += kQrThreads) {
    const int i = idx / r, k = idx % r;
    double v = 0.0;
    if (i < nrows) {
      const int64_t e = (row0 + i) * r + k;
      v = SRC_DOUBLE ? static_cast<const double*>(Xv)[e] : static_cast<double>(static_cast<const float*>(Xv)[e]);
    }
    Xs[i][k] = v;
  }
  __syncthreads();
  double* out = partials + static_cast<int64_t>(blockIdx.x) * r * r;
  for (int idx = threadIdx.x; idx < r * r; idx += kQrThreads) {
    const int a = idx / r, b = idx % r;
    double s = 0.0;
    if (b >= a) {                       // upper triangle; the factorisation reads nothing else
      for (int i = 0; i < kChunkRows; ++i) s = fma(Xs[i][a], Xs[i][b], s);
    }
    out[idx] = s;
  }
}

// S = sum of the partials (fixed order), S = R^T R, W = R^-1 (upper triangular, double, r x r row-major).
// status[0] = 0, or 1 + k if the k-th pivot is not positive (the columns of A are linearly dependent to
// working precision); W is then left unset.  If Racc is not null it is multiplied from the left by this pass's R
// (Racc <- R Racc), which after two passes is the triangular factor of A itself.
__global__ void __launch_bounds__(kQrThreads) factor_kernel(const double* __restrict__ partials, int n_chunks, int r, double* __restrict__ W,
                                                            double* __restrict__ Racc, int first_pass, int* __restrict__ status) {
  extern __shared__ double dyn_smem[];
  double (*S)[kLd] = reinterpret_cast<double (*)[kLd]>(dyn_smem);                       // [kMaxR][kLd]
  double (*Winv)[kLd] = reinterpret_cast<double (*)[kLd]>(dyn_smem + kMaxR * kLd);
  double (*Old)[kLd] = reinterpret_cast<double (*)[kLd]>(dyn_smem + 2 * kMaxR * kLd);
  __shared__ int bad;
  __shared__ double norm2[kMaxR];        // diagonal before the factorisation: the columns' squared norms
  if (threadIdx.x == 0) bad = 0;
  for (int idx = threadIdx.x; idx < r * r; idx += kQrThreads) {
    // (with the rounding errors of the additions kept and added last: 60,000 rows are 469 chunks, whose plain sum is off by as
    // much as the pivot of directions 3e-8 apart)
    double s = 0.0, lost = 0.0;
    for (int c = 0; c < n_chunks; ++c) {
      const double x = partials[static_cast<int64_t>(c) * r * r + idx], t = s + x, back = t - s;
      lost += (s - (t - back)) + (x - back);
      s = t;
    }
    s += lost;
    S[idx / r][idx % r] = s;
    if (idx / r == idx % r) norm2[idx / r] = s;
  }
  __syncthreads();
  // Cholesky, column by column (right-looking), upper triangular factor kept in the upper triangle of S
  for (int k = 0; k < r; ++k) {
    if (threadIdx.x == 0) {
      const double p = S[k][k];
      if (!(p > kPivotFloor * norm2[k]) && bad == 0) bad = 1 + k;
      S[k][k] = p > 0.0 ? sqrt(p) : 1.0;
    }
    __syncthreads();
    const double d = S[k][k];
    for (int j = k + 1 + threadIdx.x; j < r; j += kQrThreads) S[k][j] /= d;
    __syncthreads();
    for (int idx = threadIdx.x; idx < (r - k - 1) * (r - k - 1); idx += kQrThreads) {
      const int i = k + 1 + idx / (r - k - 1), j = k + 1 + idx % (r - k - 1);
      if (j >= i) S[i][j] -= S[k][i] * S[k][j];
    }
    __syncthreads();
  }
  // inverse of the upper triangular R by back substitution, one column per thread
  for (int j = threadIdx.x; j < r; j += kQrThreads) {
    for (int i = r - 1; i >= 0; --i) {
      double v = (i == j) ? 1.0 : 0.0;
      for (int k = i + 1; k <= j; ++k) v -= S[i][k] * Winv[k][j];
      Winv[i][j] = (i <= j) ? v / S[i][i] : 0.0;
    }
  }
  __syncthreads();
  for (int idx = threadIdx.x; idx < r * r; idx += kQrThreads) W[idx] = Winv[idx / r][idx % r];
  if (Racc != nullptr) {
    // Racc <- R Racc  (first pass: Racc = R)
    for (int idx = threadIdx.x; idx < r * r; idx += kQrThreads) Old[idx / r][idx % r] = first_pass ? ((idx / r == idx % r) ? 1.0 : 0.0) : Racc[idx];
    __syncthreads();
    for (int idx = threadIdx.x; idx < r * r; idx += kQrThreads) {
      const int i = idx / r, j = idx % r;
      double v = 0.0;
      for (int k = i; k <= j; ++k) v += S[i][k] * Old[k][j];
      Racc[idx] = (j >= i) ? v : 0.0;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0 && bad != 0 && status[0] == 0) status[0] = bad;
}

// Y = X W for rows [chunk*128, +128): X fp32 or double (rows x r), W double upper triangular, Y double or fp32.
template <bool SRC_DOUBLE, bool DST_DOUBLE>
__global__ void __launch_bounds__(kQrThreads) apply_kernel(const void* __restrict__ Xv, int64_t rows, int r, const double* __restrict__ W,
                                                           void* __restrict__ Yv, const int* __restrict__ status) {
  if (status[0] != 0) return;          // the factorisation failed: leave the destination alone
  extern __shared__ double dyn_smem[];
  double (*Xs)[kLd] = reinterpret_cast<double (*)[kLd]>(dyn_smem);                      // [kChunkRows][kLd]
  double (*Ws)[kLd] = reinterpret_cast<double (*)[kLd]>(dyn_smem + kChunkRows * kLd);   // [kMaxR][kLd]
  const int64_t row0 = static_cast<int64_t>(blockIdx.x) * kChunkRows;
  const int nrows = static_cast<int>(min(static_cast<int64_t>(kChunkRows), rows - row0));
  for (int idx = threadIdx.x; idx < r * r; idx += kQrThreads) Ws[idx / r][idx % r] = W[idx];
  for (int idx = threadIdx.x; idx < nrows * r; idx += kQrThreads) {
    const int i = idx / r, k = idx % r;
    const int64_t e = (row0 + i) * r + k;
    Xs[i][k] = SRC_DOUBLE ? static_cast<const double*>(Xv)[e] : static_cast<double>(static_cast<const float*>(Xv)[e]);
  }
  __syncthreads();
  for (int idx = threadIdx.x; idx < nrows * r; idx += kQrThreads) {
    const int i = idx / r, j = idx % r;
    double v = 0.0;
    for (int k = 0; k <= j; ++k) v = fma(Xs[i][k], Ws[k][j], v);
    const int64_t e = (row0 + i) * r + j;
    if (DST_DOUBLE) static_cast<double*>(Yv)[e] = v;
    else static_cast<float*>(Yv)[e] = static_cast<float>(v);
  }
}

// ---------------------------------------------------------------------------------------------
// the whole construction in one launch
// ---------------------------------------------------------------------------------------------
__host__ __device__ constexpr int cluster_ctas(int rc) { return rc == 16 ? 16 : 8; }
// Entries per CTA up to which one cluster beats the grid (cycles, cluster / grid, at twice that size: 51k / 45k at rank 16,
// 77k / 60k at rank 32, 121k / 116k at rank 64; the grid pays four barriers of 3k and two more reductions).
constexpr int kClusterEntries = 4096;
inline bool in_cluster(int64_t rows, int rc) { return (rows + cluster_ctas(rc) - 1) / cluster_ctas(rc) * rc <= (rc == 64 ? 2 : 1) * kClusterEntries; }
constexpr long long kBarrierLimit = 4000000000ll;   // cycles, about 2 s: a barrier that waits longer gives up

struct BasisArgs {
  const float* A;       // rows x r
  float* U;             // rows x r, may be A
  SplitJob copies;      // operand copies to refresh (part[0] null: none)
  double* partials;     // one RC x RC matrix per CTA (cluster launches: and pass)
  double* sum;          // RC x RC (grid launches)
  unsigned* counter;    // grid barrier: arrivals, exits, a CTA gave up; all zero between launches
  volatile int* status; // host-mapped: 0, 1 + dependent column, or -1 if a barrier gave up
  int64_t rows;
  int r;
  int rows_per_cta;
};

// 1 / x by two Newton steps on the hardware's approximation (20 bits -> 40 -> working precision): half the latency of a
// division, and the chain from column to column of the factorisation waits for it.
__device__ __forceinline__ double reciprocal(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  y = fma(fma(-x, y, 1.0), y, y);
  return fma(fma(-x, y, 1.0), y, y);
}

template <bool CLUSTER>
__device__ __forceinline__ bool basis_barrier(unsigned* counter, int index) {
  if constexpr (CLUSTER) {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    return true;
  } else {
    // barrier number `index` of this launch; the last CTA to leave puts the counter back to zero
    __shared__ int ok;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
      const unsigned target = gridDim.x * static_cast<unsigned>(index + 1);
      atomicAdd(counter, 1u);
      const long long t0 = clock64();
      unsigned seen;
      do {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(counter) : "memory");
      } while (seen < target && clock64() - t0 < kBarrierLimit);
      ok = seen >= target;
    }
    __syncthreads();
    return ok != 0;
  }
}

// The words of `counter` for leave_grid
struct ExitWords {
  unsigned* counter;
  __device__ __forceinline__ void fail() { atomicExch(counter + 2, 1u); }
  __device__ __forceinline__ bool count_out(unsigned n) {
    __threadfence();
    const bool last = atomicInc(counter + 1, n - 1) == n - 1;
    __threadfence();
    return last;
  }
  __device__ __forceinline__ bool take_failed() { return atomicExch(counter + 2, 0u) != 0; }
};

// RC = r rounded up to 16, 32 or 64.
//
// Gram matrix: groups of 64 threads take rows in turn; thread (ui, uj) of a group owns the entries (ui + 8 x, uj + 8 y),
// x <= y, which needs RC/4 shared-memory reads per (RC/8)^2 / 2 multiply-adds (one entry per thread is bound by those reads:
// 36 cycles per row at RC = 16 against 8).  The groups' sums are added in order.
// Factorisation: S = L D L^T and, by the same eliminations applied to the identity, M = L^-1; then R^-1 = M^T D^-1/2.
// Thread (ti, tj) of a 16 x 16 arrangement owns the entries (ti + 16 a, tj + 16 b): a <= b of S, a >= b of M.  One barrier per
// column; only the reciprocal of the pivot is on the chain from column to column.  (512 threads at RC = 64: 73 us a call
// instead of 58, the barriers cost more than the shorter updates save.)
// Product X R^-1: at RC = 16 a thread takes a row, otherwise a warp eight rows, a lane four of them and the columns tj + 16 b.
template <int RC, bool CLUSTER>
__global__ void __launch_bounds__(kQrThreads) basis_kernel(const BasisArgs p) {
  constexpr int kT = kQrThreads, NB = RC / 16, LD = RC + 1, CL = cluster_ctas(RC);
  extern __shared__ double dyn_smem[];
  double* Ms = dyn_smem;                       // RC x LD: rows of M (before that: the sum of the groups' Gram matrices)
  double* rowbuf = Ms + RC * LD;               // 2 x RC: current row of D L^T
  double* inv = rowbuf + 2 * RC;               // D[k], then D[k]^-1/2
  double* diag = inv + RC;                     // diagonal before the factorisation
  double* X = diag + RC;                       // rows_per_cta x LD
  const int tid = threadIdx.x, ti = tid >> 4, tj = tid & 15;
  const int64_t row0 = static_cast<int64_t>(blockIdx.x) * p.rows_per_cta;
  const int nrows = static_cast<int>(max(static_cast<int64_t>(0), min(static_cast<int64_t>(p.rows_per_cta), p.rows - row0)));
  const int r = p.r;
  int status = 0;

#pragma unroll 8
  for (int idx = tid; idx < nrows * RC; idx += kT) {
    const int i = idx / RC, k = idx % RC;
    X[i * LD + k] = k < r ? static_cast<double>(p.A[(row0 + i) * r + k]) : 0.0;
  }
  __syncthreads();

#pragma unroll 1
  for (int pass = 0; pass < 2 && status == 0; ++pass) {
    // ---- Gram matrix of this CTA's rows ----
    double s[NB][NB];
    {
      constexpr int B = RC / 8;
      const int grp = tid >> 6, ui = (tid >> 3) & 7, uj = tid & 7;
      double acc[B][B];
#pragma unroll
      for (int x = 0; x < B; ++x)
#pragma unroll
        for (int y = 0; y < B; ++y) acc[x][y] = 0.0;
#pragma unroll (RC == 64 ? 1 : 4)
      for (int i = grp; i < nrows; i += kT / 64) {
        const double* row = X + i * LD;
        double u[B], v[B];
#pragma unroll
        for (int x = 0; x < B; ++x) { u[x] = row[ui + 8 * x]; v[x] = row[uj + 8 * x]; }
#pragma unroll
        for (int x = 0; x < B; ++x)
#pragma unroll
          for (int y = x; y < B; ++y) acc[x][y] = fma(u[x], v[y], acc[x][y]);
      }
#pragma unroll 1
      for (int g = 0; g < kT / 64; ++g) {
        if (grp == g) {
#pragma unroll
          for (int x = 0; x < B; ++x)
#pragma unroll
            for (int y = x; y < B; ++y) {
              double* at = Ms + (ui + 8 * x) * RC + uj + 8 * y;
              *at = g == 0 ? acc[x][y] : *at + acc[x][y];
            }
        }
        __syncthreads();
      }
      // (a cluster has one barrier per pass, so the second pass writes its own set)
      double* out = p.partials + static_cast<int64_t>(blockIdx.x + (CLUSTER ? pass * CL : 0)) * RC * RC;
#pragma unroll
      for (int a = 0; a < NB; ++a)
#pragma unroll
        for (int b = a; b < NB; ++b) {
          const int i = ti + 16 * a, j = tj + 16 * b;
          out[i * RC + j] = Ms[min(i, j) * RC + max(i, j)];
        }
    }
    if (!basis_barrier<CLUSTER>(p.counter, 2 * pass)) { status = -1; break; }
    // ---- their sum, in a fixed order ----
    if constexpr (CLUSTER) {
#pragma unroll
      for (int a = 0; a < NB; ++a)
#pragma unroll
        for (int b = a; b < NB; ++b) {
          double v = 0.0;
#pragma unroll
          for (int c = 0; c < CL; ++c)
            v += __ldcg(p.partials + static_cast<int64_t>(c + pass * CL) * RC * RC + (ti + 16 * a) * RC + tj + 16 * b);
          s[a][b] = v;
        }
    } else {
      // a warp per entry, four entries at a time (entries of the blocks below the diagonal hold nothing and go unused)
      const int lane = tid & 31, wid = blockIdx.x * (kT / 32) + (tid >> 5), warps = static_cast<int>(gridDim.x) * (kT / 32);
      for (int e0 = wid; e0 < RC * RC; e0 += 4 * warps) {
        double v[4] = {0.0, 0.0, 0.0, 0.0};
        for (int c = lane; c < static_cast<int>(gridDim.x); c += 32) {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int e = e0 + q * warps;
            if (e < RC * RC && (e / RC) / 16 <= (e % RC) / 16) v[q] += __ldcg(p.partials + static_cast<int64_t>(c) * RC * RC + e);
          }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1)
#pragma unroll
          for (int q = 0; q < 4; ++q) v[q] += __shfl_xor_sync(0xFFFFFFFFu, v[q], off);
        if (lane == 0) {
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (e0 + q * warps < RC * RC) p.sum[e0 + q * warps] = v[q];
        }
      }
      if (!basis_barrier<CLUSTER>(p.counter, 2 * pass + 1)) { status = -1; break; }
#pragma unroll
      for (int a = 0; a < NB; ++a)
#pragma unroll
        for (int b = a; b < NB; ++b) s[a][b] = __ldcg(p.sum + (ti + 16 * a) * RC + tj + 16 * b);
    }
    // ---- S = L D L^T, M = L^-1 ----
    double m[NB][NB];
#pragma unroll
    for (int a = 0; a < NB; ++a)
#pragma unroll
      for (int b = 0; b <= a; ++b) {
        const bool on_diagonal = a == b && ti == tj;
        m[a][b] = on_diagonal ? 1.0 : 0.0;
        if (on_diagonal) diag[ti + 16 * a] = s[a][a];
      }
#pragma unroll
    for (int a = 0; a < NB; ++a) {
      const int kk_end = min(16, r - 16 * a);
#pragma unroll 1
      for (int kk = 0; kk < kk_end; ++kk) {
        const int k = 16 * a + kk;
        double* row = rowbuf + (k & 1) * RC;
        if (ti == kk) {
#pragma unroll
          for (int b = a; b < NB; ++b) row[tj + 16 * b] = s[a][b];
#pragma unroll
          for (int b = 0; b <= a; ++b) Ms[k * LD + tj + 16 * b] = m[a][b];
        }
        __syncthreads();
        const double piv = row[k];
        if (status == 0 && !(piv > kPivotFloor * diag[k])) status = 1 + k;      // the same decision in every thread of every CTA
        const double ip = reciprocal(piv);
        if (tid == k) inv[k] = piv;
#pragma unroll
        for (int a2 = a; a2 < NB; ++a2) {
          const int i = ti + 16 * a2;
          if (i > k) {
            const double f = row[i] * ip;
#pragma unroll
            for (int b2 = a2; b2 < NB; ++b2) s[a2][b2] = fma(-f, row[tj + 16 * b2], s[a2][b2]);
#pragma unroll
            for (int b2 = 0; b2 <= a; ++b2) m[a2][b2] = fma(-f, Ms[k * LD + tj + 16 * b2], m[a2][b2]);
          }
        }
      }
    }
    __syncthreads();
    if (status != 0) break;
    if (pass == 0) {
      // Is the second pass needed (see kOnePass)?  sum_k |a_k|^2 (R^-1)_kj^2 for every column j, by the 16 threads that hold row j of M.
      bool again = false;
#pragma unroll
      for (int a = 0; a < NB; ++a) {
        double v = 0.0;
#pragma unroll
        for (int b = 0; b <= a; ++b) v = fma(diag[tj + 16 * b] * m[a][b], m[a][b], v);
#pragma unroll
        for (int off = 8; off > 0; off >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, off);
        if (ti + 16 * a < r && !(v * r <= kOnePass * inv[ti + 16 * a])) again = true;
      }
      if (!__syncthreads_or(again)) pass = 1;      // (the same answer in every CTA: all have the same sums)
    }
    if (tid < RC) inv[tid] = tid < r ? 1.0 / sqrt(inv[tid]) : 0.0;
    for (int idx = tid; idx < (RC - r) * RC; idx += kT) Ms[(r + idx / RC) * LD + idx % RC] = 0.0;      // rank not a multiple of 16
    __syncthreads();
    // ---- X <- X R^-1 = X M^T D^-1/2 ----
    if constexpr (RC == 16) {
      // one row per thread: 136 broadcast reads and as many multiply-adds
      for (int i = tid; i < nrows; i += kT) {
        double* xr = X + i * LD;
        asm volatile("" ::: "memory");      // M stays in shared memory: hoisted out of the row loop it would fill the register file
        double x[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) x[k] = xr[k];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          double q = 0.0;
#pragma unroll
          for (int k = 0; k <= j; ++k) q = fma(x[k], Ms[j * LD + k], q);
          xr[j] = q * inv[j];
        }
      }
    } else {
      const int warp = tid >> 5, half = (tid >> 4) & 1;
#pragma unroll 1
      for (int i0 = 8 * warp; i0 < nrows; i0 += kT / 4) {
        const int i1 = i0 + 4 * half;
        const double* xr[4];
        double q[4][NB];
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          xr[h] = X + min(i1 + h, nrows - 1) * LD;
#pragma unroll
          for (int b = 0; b < NB; ++b) q[h][b] = 0.0;
        }
#pragma unroll
        for (int kb = 0; kb < NB; ++kb) {
#pragma unroll 4
          for (int kk = 0; kk < 16; ++kk) {
            const int k = 16 * kb + kk;
            double x[4];
#pragma unroll
            for (int h = 0; h < 4; ++h) x[h] = xr[h][k];
#pragma unroll
            for (int b = kb; b < NB; ++b) {
              const int j = tj + 16 * b;
              const double w = (b > kb || k <= j) ? Ms[j * LD + k] : 0.0;
#pragma unroll
              for (int h = 0; h < 4; ++h) q[h][b] = fma(x[h], w, q[h][b]);
            }
          }
        }
        __syncwarp();
#pragma unroll
        for (int h = 0; h < 4; ++h)
          if (i1 + h < nrows) {
#pragma unroll
            for (int b = 0; b < NB; ++b) X[(i1 + h) * LD + tj + 16 * b] = q[h][b] * inv[tj + 16 * b];
          }
        __syncwarp();
      }
    }
    __syncthreads();
  }

  if (status == 0) {
    const SplitJob& c = p.copies;
    const float scale = c.shift >= 0 ? __int_as_float((127 + c.shift) << 23) : 1.0f;
#pragma unroll 4
    for (int idx = tid; idx < nrows * RC; idx += kT) {
      const int i = idx / RC, k = idx % RC;
      if (k >= r) continue;                    // (the padding of the copies is zero since zgr_init)
      const float u = static_cast<float>(X[i * LD + k]);
      p.U[(row0 + i) * r + k] = u;
      if (c.part[0] != nullptr) split_subspace_entry(c, row0 + i, k, u, scale);
    }
  }
  // The host polls the status word: it is written once every CTA's results are visible.
  __threadfence();
  if constexpr (CLUSTER) {
    basis_barrier<CLUSTER>(p.counter, 0);
    if (blockIdx.x == 0 && tid == 0) {
      __threadfence_system();
      *p.status = status;
    }
  } else {
    __syncthreads();
    ExitWords words{p.counter};
    if (tid == 0 && leave_grid(words, gridDim.x, status)) {
      *p.counter = 0;
      __threadfence_system();
      *p.status = status;
    }
  }
}

template <int RC>
size_t basis_smem(int rows_per_cta) {
  return (static_cast<size_t>(RC) * (RC + 1) + 4 * RC + static_cast<size_t>(rows_per_cta) * (RC + 1)) * sizeof(double);
}
constexpr size_t kBasisSmemMax = 232448 - 1024;

template <int RC>
cudaError_t launch_basis(BasisArgs p, int sm_count, cudaStream_t st, bool* served) {
  *served = true;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  cfg.blockDim = dim3(kQrThreads);
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  constexpr int CL = cluster_ctas(RC);
  if (in_cluster(p.rows, RC)) {
    p.rows_per_cta = static_cast<int>((p.rows + CL - 1) / CL);
    const size_t smem = basis_smem<RC>(p.rows_per_cta);
    cudaError_t e = cudaFuncSetAttribute(basis_kernel<RC, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kBasisSmemMax));
    if (e == cudaSuccess && CL > 8) e = cudaFuncSetAttribute(basis_kernel<RC, true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cfg.gridDim = dim3(CL);
    cfg.dynamicSmemBytes = smem;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CL;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    return cudaLaunchKernelEx(&cfg, basis_kernel<RC, true>, p);
  }
  const int64_t per_cta = std::max<int64_t>((p.rows + sm_count - 1) / sm_count, 64);
  if (per_cta > (1 << 20) || basis_smem<RC>(static_cast<int>(per_cta)) > kBasisSmemMax) {
    *served = false;
    return cudaSuccess;
  }
  p.rows_per_cta = static_cast<int>(per_cta);
  const cudaError_t e = cudaFuncSetAttribute(basis_kernel<RC, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kBasisSmemMax));
  if (e != cudaSuccess) return e;
  cfg.gridDim = dim3(static_cast<unsigned>((p.rows + per_cta - 1) / per_cta));
  cfg.dynamicSmemBytes = basis_smem<RC>(p.rows_per_cta);
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  return cudaLaunchKernelEx(&cfg, basis_kernel<RC, false>, p);
}

}  // namespace

// Scratch layout: [0, 256) status of the three-kernel path, [256, 512) barrier counter, then the matrices.
size_t subspace_scratch_bytes(int64_t rows, int r, int sm_count) {
  const int64_t n_chunks = (rows + kChunkRows - 1) / kChunkRows;
  // three-kernel path: partial Gram matrices, R^-1, accumulated R, the double image of the first pass's Q
  const size_t chunked = static_cast<size_t>(n_chunks) * r * r * sizeof(double) + 2 * static_cast<size_t>(r) * r * sizeof(double) +
                         static_cast<size_t>(rows) * r * sizeof(double);
  const int rc = r <= 16 ? 16 : (r <= 32 ? 32 : 64);
  const size_t matrices = 1 + static_cast<size_t>(in_cluster(rows, rc) ? 2 * cluster_ctas(rc) : sm_count);
  const size_t fused = matrices * static_cast<size_t>(rc * rc) * sizeof(double);
  return 512 + (subspace_fused(rows, r, sm_count) ? fused : chunked);
}

bool subspace_fused(int64_t rows, int r, int sm_count) {
  const int64_t per_cta = std::max<int64_t>((rows + sm_count - 1) / sm_count, 64);
  if (per_cta > (1 << 20)) return false;
  const int n = static_cast<int>(per_cta);
  return (r <= 16 ? basis_smem<16>(n) : (r <= 32 ? basis_smem<32>(n) : basis_smem<64>(n))) <= kBasisSmemMax;
}

cudaError_t launch_basis_fused(const float* A, int64_t rows, int r, float* U_out, const SplitJob* copies, void* scratch, int* status, int sm_count,
                               cudaStream_t st) {
  if (r < 1 || r > kMaxR || rows < r) return cudaErrorInvalidValue;
  BasisArgs p = {};
  p.A = A;
  p.U = U_out;
  if (copies) p.copies = *copies;
  uint8_t* base = static_cast<uint8_t*>(scratch);
  p.counter = reinterpret_cast<unsigned*>(base + 256);
  const int rc = r <= 16 ? 16 : (r <= 32 ? 32 : 64);
  p.sum = reinterpret_cast<double*>(base + 512);
  p.partials = p.sum + rc * rc;
  p.status = status;
  p.rows = rows;
  p.r = r;
  bool served = false;
  const cudaError_t e = rc == 16 ? launch_basis<16>(p, sm_count, st, &served)
                                 : (rc == 32 ? launch_basis<32>(p, sm_count, st, &served) : launch_basis<64>(p, sm_count, st, &served));
  return e == cudaSuccess && !served ? cudaErrorInvalidValue : e;
}

cudaError_t launch_build_subspace(const float* A, int64_t rows, int r, float* U_out, void* scratch, int** status_out, double** r_out, cudaStream_t st) {
  if (r < 1 || r > kMaxR || rows < r) return cudaErrorInvalidValue;
  const int n_chunks = static_cast<int>((rows + kChunkRows - 1) / kChunkRows);
  uint8_t* base = static_cast<uint8_t*>(scratch);
  int* status = reinterpret_cast<int*>(base);
  double* partials = reinterpret_cast<double*>(base + 512);
  double* W = partials + static_cast<size_t>(n_chunks) * r * r;
  double* Racc = W + static_cast<size_t>(r) * r;
  double* Q1 = Racc + static_cast<size_t>(r) * r;
  constexpr int kGramSmem = kChunkRows * kLd * sizeof(double);
  constexpr int kFactorSmem = 3 * kMaxR * kLd * sizeof(double);
  constexpr int kApplySmem = (kChunkRows + kMaxR) * kLd * sizeof(double);
  // (on every call: the attributes belong to the current device, and a context may live on any)
  cudaError_t e = cudaFuncSetAttribute(gram_partial_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kGramSmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(gram_partial_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kGramSmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(factor_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kFactorSmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(apply_kernel<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kApplySmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(apply_kernel<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kApplySmem);
  if (e == cudaSuccess) e = cudaMemsetAsync(status, 0, sizeof(int), st);
  if (e != cudaSuccess) return e;
  // pass 1: A (fp32) -> Q1 (double)
  gram_partial_kernel<false><<<n_chunks, kQrThreads, kGramSmem, st>>>(A, rows, r, partials);
  factor_kernel<<<1, kQrThreads, kFactorSmem, st>>>(partials, n_chunks, r, W, Racc, 1, status);
  apply_kernel<false, true><<<n_chunks, kQrThreads, kApplySmem, st>>>(A, rows, r, W, Q1, status);
  // pass 2: Q1 (double) -> U (fp32)
  gram_partial_kernel<true><<<n_chunks, kQrThreads, kGramSmem, st>>>(Q1, rows, r, partials);
  factor_kernel<<<1, kQrThreads, kFactorSmem, st>>>(partials, n_chunks, r, W, Racc, 0, status);
  apply_kernel<true, false><<<n_chunks, kQrThreads, kApplySmem, st>>>(Q1, rows, r, W, U_out, status);
  if (status_out) *status_out = status;
  if (r_out) *r_out = Racc;
  return cudaGetLastError();
}

}  // namespace zgr
