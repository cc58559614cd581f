// The coefficient strip of the kernels that contract three bf16 parts per operand (zgr_staged.cu, zgr_tile.cu).
#ifndef ZGR_STRIP_CUH_
#define ZGR_STRIP_CUH_

#include "zgr_device.cuh"
#include "zgr_kernels.h"
#include "zgr_tcgen05.cuh"

namespace zgr {

constexpr int kTileN = 144;                    // widest strip: 128 columns and the 16 that its octets may reach into
constexpr int kEpi = 16;                       // epilogue warps
constexpr int kParts = 3;                      // bf16 parts of an operand

__device__ __forceinline__ void sts16(uint32_t saddr, uint16_t v) { asm volatile("st.shared.b16 [%0], %1;" ::"r"(saddr), "h"(v) : "memory"); }

// Compressed coefficient of row k, column c, before scale and zero point.
__device__ __forceinline__ float code1(const TensorDesc& td, int k, int64_t c) {
  if (td.qbits == 4) {
    const uint32_t byte = reinterpret_cast<const uint8_t*>(td.q)[static_cast<int64_t>(k) * ((td.cols + 1) >> 1) + (c >> 1)];
    return static_cast<float>((c & 1) ? (byte >> 4) : (byte & 15u));
  }
  return static_cast<float>(td.q[static_cast<int64_t>(k) * td.cols + c]);
}

// The strip  c b G[0..KP)[col0 .. col0 + width)  as K-major bf16 operands, by the kEpi epilogue warps (et: thread among them); width =
// 128, or 144 where octets reach beyond the strip.  One unit of work is the octet of one row k of G (the octets of G start at
// other columns in every row when cols is no multiple of 8).
template <int BITS, bool PRECISE, bool MULTI>
__device__ __forceinline__ void build_strip(const TensorDesc& td, const SweepParams& p, int64_t col0, int width, int kp, int rowb, int g_bytes, uint32_t g_dst,
                                            int et) {
  const int kp_shift = kp == 64 ? 6 : (kp == 32 ? 5 : 4);
  const int64_t cols = td.cols;
  const int n_oct = width == kTileN || (cols & 7) != 0 ? width / 8 + 1 : width / 8;      // (a constant in the tile kernel)
  for (int idx = et; idx < (n_oct << kp_shift); idx += kEpi * 32) {
    const int k = idx & (kp - 1), o = idx >> kp_shift;      // consecutive lanes: consecutive k, i.e. neighbouring shared-memory words
    const int64_t row_e = static_cast<int64_t>(k) * cols;
    const int64_t e = (((row_e + col0) >> 3) + o) << 3;     // first element of the octet
    const int64_t c_first = e - row_e;                      // its column (may lie before the strip)
    const int j0 = static_cast<int>(c_first - col0);        // -7 .. width
    float g[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) g[i] = 0.0f;
    if (k < td.rank && c_first < cols) {
      if (td.q != nullptr && k < td.qrows && (cols & 7) == 0) {
        guided8<BITS, PRECISE, MULTI>(td, p, k, c_first, g);      // eight codes of one row in one load
      } else if (td.q != nullptr && k < td.qrows) {
        float cb = p.term[0].cb;
        if (MULTI)
          for (int q = 1; q < p.n_terms; ++q) cb += p.term[q].cb;
        const float lambda = td.qscale[k] * cb;
        const float delta = td.qzero ? td.qzero[k] : 0.0f;
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (c_first + i >= 0 && c_first + i < cols) g[i] = lambda * (code1(td, k, c_first + i) - delta);
      } else {
        normals8<BITS, PRECISE>(p.term[0].keys, static_cast<uint32_t>(td.id), 1u, static_cast<uint64_t>(e), p.unit, g);
#pragma unroll
        for (int i = 0; i < 8; ++i) g[i] *= p.term[0].cb;
        if (MULTI) {
#pragma unroll 1
          for (int q = 1; q < p.n_terms; ++q) {
            float y[8];
            normals8<BITS, PRECISE>(p.term[q].keys, static_cast<uint32_t>(td.id), 1u, static_cast<uint64_t>(e), p.unit, y);
#pragma unroll
            for (int i = 0; i < 8; ++i) g[i] = fmaf(p.term[q].cb, y[i], g[i]);
          }
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int j = j0 + i;
      if (j >= 0 && j < width) {
        uint16_t q0, q1, q2;
        split_subspace_value(false, c_first + i < cols ? g[i] : 0.0f, 1.0f, 0.0f, q0, q1, q2);
        const uint32_t at = g_dst + swizzle(static_cast<uint32_t>(j * rowb + 2 * k), rowb);
        sts16(at, q0);
        sts16(at + g_bytes, q1);
        sts16(at + 2 * g_bytes, q2);
      }
    }
  }
}

}  // namespace zgr
#endif  // ZGR_STRIP_CUH_
