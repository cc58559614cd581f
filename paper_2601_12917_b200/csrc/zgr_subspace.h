// Launchers of the subspace construction kernels (Cholesky QR applied twice, carried in double).
#ifndef ZGR_SUBSPACE_H_
#define ZGR_SUBSPACE_H_

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "zgr_kernels.h"

namespace zgr {

// Bytes of device scratch that the construction needs for a rows x r input.  The first 512 bytes must be zero before the
// first launch that uses the scratch.
size_t subspace_scratch_bytes(int64_t rows, int r, int sm_count);

// Orthonormal basis of the span of the columns of A (device, rows x r fp32 row-major, r <= 64, rows >= r) into
// U_out (device, rows x r fp32 row-major; may be A itself), and its operand copies as `copies` lays them out (null:
// none), in one launch on `st`.  *status (host memory mapped into the device) is 0 afterwards, 1 + k if the k-th column of A
// depends linearly on the earlier ones to working precision (nothing is written then), or -1 if a barrier gave up.
// Serves the inputs that subspace_fused says yes to.
bool subspace_fused(int64_t rows, int r, int sm_count);
cudaError_t launch_basis_fused(const float* A, int64_t rows, int r, float* U_out, const SplitJob* copies, void* scratch, int* status, int sm_count,
                               cudaStream_t st);

// The same for larger inputs, in six launches and without the operand copies.  *status_out (if not null) receives the device
// address of the status.  *r_out (if not null) receives the device address of the triangular factor R (r x r doubles,
// row-major, A = U R, positive diagonal).
cudaError_t launch_build_subspace(const float* A, int64_t rows, int r, float* U_out, void* scratch, int** status_out, double** r_out, cudaStream_t st);

}  // namespace zgr
#endif  // ZGR_SUBSPACE_H_
