// Host-visible launchers of the sweep kernels.
#ifndef ZGR_KERNELS_H_
#define ZGR_KERNELS_H_

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stddef.h>

#include "zgr.h"
#include "zgr_internal.h"

namespace zgr {

enum Path { PATH_ISO = 0, PATH_FMA = 1, PATH_MMA = 2, PATH_GENERIC = 3, PATH_UMMA = 4, PATH_COUNT = 5 };

// Which kernel instantiation a group of work items runs on.
struct KernelChoice {
  int path;   // Path
  int dtype;  // ZGR_F32 | ZGR_F16 | ZGR_BF16
  int kpad;   // contraction width.  FMA: 4 or 8;  MMA, UMMA and the three-part kernels (see is_tile): 16, 32 or 64;  otherwise 0
  int bits;   // 32 or 16 random bits per normal
  int precise;  // accurate Gaussian transform (tensors stored in fp32)
  int staged;   // among the groups of is_tile: served by sweep_staged_kernel
  int by_residue;  // tile kernel: copies of U in the order of staged_copy_row, behind 4-D maps
};

// Resident blocks of 256 threads per SM of the isotropic kernel.  Its plain instantiation (fused transform) fits 32 registers:
// eight blocks, whose loads then cover the DRAM latency (5.74 TB/s standalone against 5.50 with six).
constexpr int iso_blocks_per_sm(bool precise, bool multi, bool stats) { return !precise && !multi && !stats ? 8 : 5; }

// The groups that sweep_staged_kernel and sweep_tile_kernel serve: rank <= 8 tensors in whole octets are counted under the path of the CUDA-core
// kernel (whose own widths are 4 and 8), the others under that of the fallback kernel (whose own width is 0).
inline bool is_tile(const KernelChoice& kc) { return (kc.path == PATH_FMA && kc.kpad == 16) || (kc.path == PATH_GENERIC && kc.kpad > 0); }
// ZGR_KERNEL_*: the paths, and behind them the two kernels that share paths with others
inline int kernel_number(const KernelChoice& kc) { return is_tile(kc) ? (kc.staged ? ZGR_KERNEL_STAGED : ZGR_KERNEL_TILE) : kc.path; }

int mma_strip_cols(int kpad);     // columns of a CTA strip on the tensor-core path
int mma_rows_per_iter(int kpad);  // rows a CTA advances per iteration there
size_t mma_smem_bytes(int kpad);

// Launch of a kernel that handles programmatic dependencies (dependency_begin): it may start before the
// kernel ahead of it in the stream has completed.
template <typename... Params, typename... Args>
cudaError_t launch_sweep_kernel(void (*kernel)(Params...), int grid, int threads, size_t smem, cudaStream_t st, const Args&... args) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = dim3(static_cast<unsigned>(grid));
  cfg.blockDim = dim3(static_cast<unsigned>(threads));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}

cudaError_t launch_sweep(const KernelChoice& kc, const SweepParams& p, int grid, cudaStream_t st);
// tcgen05 + TMA sweep (16-bit weights, rank > 8).  tmaps: three tensor maps per tensor (theta, U hi, U lo).
int umma_strip_cols(int kpad);
size_t umma_smem_bytes(int kpad);
cudaError_t launch_sweep_umma(const KernelChoice& kc, const SweepParams& p, const CUtensorMap* tmaps, int* error, int grid, cudaStream_t st);
// Test hook: the sweep kernel with its fp32 results diverted to p.zout (see the ZOUT parameter of the kernel).
cudaError_t launch_debug_z_umma(const KernelChoice& kc, const SweepParams& p, const CUtensorMap* tmaps, int* error, int grid, cudaStream_t st);
cudaError_t launch_stats_umma(const KernelChoice& kc, const SweepParams& p, const CUtensorMap* tmaps, int* error, int grid, cudaStream_t st);
// Sweep of the other guided tensors that a tensor-core kernel serves (fp32, rank <= 8, rows that are not a multiple of eight
// elements).  kc.kpad = contraction width; strips of 128 columns.  The tile kernel takes those that TMA cannot address and small sets; tmaps: the three
// bf16 parts of U per tensor.
constexpr int kTileStripCols = 128;
cudaError_t launch_sweep_staged(const KernelChoice& kc, const SweepParams& p, int* error, int grid, cudaStream_t st);
cudaError_t launch_sweep_tile(const KernelChoice& kc, const SweepParams& p, const CUtensorMap* tmaps, int* error, int grid, cudaStream_t st);
// Rebuild of the row-major operand copies of U for a device-resident list of tensors in one launch (grid.y = job).
struct SplitJob {
  const float* U;
  void* part[3];   // rows_pad x kp each
  int64_t rows, rows_pad;
  int32_t r, kp;
  int32_t shift;   // two fp16 parts (hi, lo) of U * 2^shift; -1: three bf16 parts of U
  int32_t by_residue;  // rows in the order of staged_copy_row (tensors of sweep_staged_kernel whose rows are no multiple of eight elements)
};
// Where row m of U is kept so that the 32 rows of a quarter of a tile, m mod 8 the same, follow one another; and the row kept at c.
// (rows in spans of 256: eight residues x 32 rows)
__host__ __device__ inline int64_t staged_copy_row(int64_t m) { return (m & ~int64_t{255}) | ((m & 7) << 5) | ((m >> 3) & 31); }
__host__ __device__ inline int64_t staged_row_at(int64_t c) { return (c & ~int64_t{255}) | ((c & 31) << 3) | ((c >> 5) & 7); }
#ifdef __CUDACC__
// The parts of one entry x of U: fp16 hi + lo of x 2^shift (22 significant bits as long as the scaled entry is not far below 1:
// lo must stay a normal fp16 number), or three bf16 parts whose sum is x (1 + lean).
__device__ __forceinline__ void split_subspace_value(bool fp16, float x, float scale, float lean, uint16_t& p0, uint16_t& p1, uint16_t& p2) {
  if (fp16) {
    const float y = x * scale;                       // power of two: exact
    const __half hi = __float2half_rn(y);
    p0 = __half_as_ushort(hi);
    p1 = __half_as_ushort(__float2half_rn(y - __half2float(hi)));
    p2 = 0;
  } else {
    const __nv_bfloat16 a = __float2bfloat16_rn(x);
    const float r1 = x - __bfloat162float(a);
    const __nv_bfloat16 b = __float2bfloat16_rn(r1);
    p0 = __bfloat16_as_ushort(a);
    p1 = __bfloat16_as_ushort(b);
    p2 = __bfloat16_as_ushort(__float2bfloat16_rn(fmaf(x, lean, r1 - __bfloat162float(b))));
  }
}
// The tensor cores add towards zero: products of six parts over a contraction width of 16, 32 and 64 come out 3.0e-8, 3.8e-8 and 5.4e-8
// of themselves too small.  The third part of U makes up for it.  2-norm of the error against 64 bits, of the result's, without /
// with it / of a chain of fp32 multiply-adds:  rank 4 4.6 / 2.9 / 4.0e-8,  16 4.8 / 3.0 / 7.6e-8,  64 7.7 / 4.9 / 14.7e-8.
__device__ __forceinline__ float truncation_lean(int kp) { return 2.2e-8f + 5e-10f * static_cast<float>(kp); }
// Entry (row, k) of the copies of job j from the value x of U; scale = 2^shift.
__device__ __forceinline__ void split_subspace_entry(const SplitJob& j, int64_t row, int k, float x, float scale) {
  const int64_t at = (j.by_residue ? staged_copy_row(row) : row) * j.kp + k;
  uint16_t p0, p1, p2;
  split_subspace_value(j.shift >= 0, x, scale, truncation_lean(j.kp), p0, p1, p2);
  static_cast<uint16_t*>(j.part[0])[at] = p0;
  static_cast<uint16_t*>(j.part[1])[at] = p1;
  if (j.shift < 0) static_cast<uint16_t*>(j.part[2])[at] = p2;
}
#endif
// max_entries: rows_pad * kp of the largest of the jobs
cudaError_t launch_split_subspaces(const SplitJob* d_jobs, int n_jobs, int64_t max_entries, cudaStream_t st);

cudaError_t launch_stats(int bits, const SweepParams& p, int grid, cudaStream_t st);
// Norm bookkeeping, second stage: tensor l owns the work items [first, first + count) of the slot array `slots`
// (kStatSlots x 3 doubles per item); out[3 l + j] receives their sum, added in a fixed order.
struct StatRange {
  const double* slots;
  int32_t first, count;
};
cudaError_t launch_stats_finish(const StatRange* d_ranges, int n_tensors, double* d_out, cudaStream_t st);
cudaError_t launch_split_subspace(const float* U, int64_t rows, int r, int kp, uint4* out, cudaStream_t st);
cudaError_t launch_philox_blocks(const PhiloxKeys& keys, uint32_t tensor, uint32_t tag, uint64_t first_block, int64_t n_blocks,
                                 uint32_t* out, cudaStream_t st);

}  // namespace zgr
#endif  // ZGR_KERNELS_H_
