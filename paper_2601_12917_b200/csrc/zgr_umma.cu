// Blackwell-native sweep for 16-bit weights with a rank > 8 subspace:
//     theta <- rnd(theta + c (a Z + b U G))            (Eq. (perturbation) applied as in Algorithm 1)
//
// The generator and the Gaussian transform are most of what an SM has to issue at the rate HBM can feed the weights (the whole
// kernel issues in 55 % of the cycles, special functions fill 63 % of their pipe at rank 16), so everything else is taken out of
// the SM's instruction stream:
//
//   * TMA brings a 128-row x NS-column tile of theta (and the matching 128 x KP tiles of U, pre-split
//     into fp16 hi/lo) into shared memory, and writes the finished tile back; no thread issues a
//     global load or store for the weights.
//   * tcgen05.mma builds   D = theta + c b U G   in tensor memory (fp32):
//       - "theta" enters through identity products  D[:, 16j:16j+16] = theta[:, 16j:16j+16] * I16
//         with theta's own 16-bit tile as the A operand, which unpacks it to fp32 exactly, for free;
//       - U G is formed first, as  Ulo Ghi + Uhi Glo + Uhi Ghi  with fp16 split operands (hi + lo carries 22
//         significant bits, against 16 for a bf16 split, whose representation error of 4.5e-6 relative was the
//         whole error of z on this path).  fp16 has a narrow exponent range, so both operands are kept near 1
//         by powers of two: the library's copy of U holds U 2^j (j from the tensor's row count), the strips hold
//         c b G 2^(s-j), and the accumulator therefore holds 2^s c b U G.  The identity products that bring
//         theta in come last and use the instruction's accumulator scaling,  D <- theta I + 2^-s D
//         (s <= 15 is an immediate of the instruction), which removes the factor exactly and for free.
//         The strips of c b G live in shared memory as the K-major B operand for all row tiles of a work item.
//   * The epilogue warps, in two groups that take alternate tiles (32 rows x 64 columns per warp, 32 columns
//     at a time), read D with tcgen05.ld (one row per thread), add the isotropic
//     normals (Philox4x32-10 + Box-Muller in registers), round to the storage type and write the
//     tile into the shared-memory buffer the TMA store reads.
//
// Warp roles: warp 0 = TMA producer (loads and stores), warp 1 = MMA issuer and owner of the tensor
// memory allocation, warps 2.. = epilogue.  The two single-thread roles run in the lane picked by
// elect.sync, which lets their loop state and descriptors live in uniform registers.  One CTA per SM
// (the shared-memory footprint enforces it), persistent over its work items: a contiguous share of small sets, every
// gridDim.x-th item of the others.
//
// Every wait on an mbarrier is bounded: when a wait gives up it records where in *p.error, raises a
// CTA-wide abort flag, and all roles fall through to the common exit, where the producer drains its
// outstanding copies and warp 1 returns the tensor memory.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "zgr_device.cuh"
#include "zgr_kernels.h"
#include "zgr_tcgen05.cuh"

namespace zgr {
namespace {

constexpr unsigned kStaggerNs = 800;

template <typename T>
struct Pack16;
template <>
struct Pack16<__nv_bfloat16> {
  static constexpr int kFmt = 1;
  static constexpr uint16_t kOne = 0x3F80;
  static __device__ __forceinline__ uint32_t pack(float a, float b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&h);
  }
};
template <>
struct Pack16<__half> {
  static constexpr int kFmt = 0;
  static constexpr uint16_t kOne = 0x3C00;
  static __device__ __forceinline__ uint32_t pack(float a, float b) {
    const __half2 h = __floats2half2_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&h);
  }
};

// the eight 16-bit values of a 16-byte chunk as floats
template <typename T>
__device__ __forceinline__ void unpack8(const uint4& raw, float (&v)[8]) {
  const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if constexpr (sizeof(T) == 2 && Pack16<T>::kFmt == 1) {
      v[2 * i] = __uint_as_float(w[i] << 16);
      v[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
    } else {
      const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[i]));
      v[2 * i] = f.x;
      v[2 * i + 1] = f.y;
    }
  }
}
// fp16 hi/lo split of a pair of floats, packed as f16x2 (first value in the low half)
__device__ __forceinline__ void split_f16(float x0, float x1, uint32_t& hi, uint32_t& lo) {
  const __half2 h = __floats2half2_rn(x0, x1);
  hi = *reinterpret_cast<const uint32_t*>(&h);
  const float2 hf = __half22float2(h);
  const __half2 l = __floats2half2_rn(x0 - hf.x, x1 - hf.y);
  lo = *reinterpret_cast<const uint32_t*>(&l);
}

// Accumulator scale of a tensor in this call: s = clamp(ushift + kshift, 0, 15) (see the operand precision note above)
__device__ __forceinline__ int acc_shift(const TensorDesc& td, const SweepParams& p) { return min(max(td.ushift + p.kshift, 0), 15); }

// Tile configuration per contraction width: compile-time parameters (-D...) whose defaults are the measured
// optimum on B200.  TILE_N = 192 runs 24 epilogue warps on 128 x 192 tiles (three 64-column boxes);
// TILE_N = 128 runs 16 on 128 x 128 tiles.  S = theta stages, N = adjacent tiles per strip.
#ifndef ZGR_TILE_N16
#define ZGR_TILE_N16 128
#endif
#ifndef ZGR_TILE_N32
#define ZGR_TILE_N32 128
#endif
#ifndef ZGR_S16
#define ZGR_S16 6
#endif
#ifndef ZGR_S32
#define ZGR_S32 5
#endif
#ifndef ZGR_S64
#define ZGR_S64 4
#endif
#ifndef ZGR_N16
#define ZGR_N16 2
#endif
#ifndef ZGR_N32
#define ZGR_N32 2
#endif
#ifndef ZGR_N64
#define ZGR_N64 1
#endif
// Epilogue groups: 1 = every epilogue warp works on every tile (32 rows x 32 columns each); 2 (4) = two (four)
// groups of warps take tiles in turn (32 rows x 64 (128) columns each, in two (four) passes), so that one group's
// per-tile waits fall under the other groups' arithmetic.
#ifndef ZGR_GROUPS
#define ZGR_GROUPS 2
#endif
template <int KP>
struct UmmaCfg {
  static constexpr int NS = KP == 64 ? 128 : (KP == 32 ? ZGR_TILE_N32 : ZGR_TILE_N16);   // columns per tile / per accumulator buffer
  static constexpr bool WIDE = NS > 128;
  static constexpr int EPI_WARPS = NS / 8;                 // one epilogue warp per 32 rows x 32 columns of a tile
  static constexpr int THREADS = 32 * (2 + EPI_WARPS);
  static constexpr int GROUPS = NS == 128 ? ZGR_GROUPS : 1;   // epilogue groups on alternate tiles (1, 2 or 4; see ZGR_GROUPS)
  static constexpr int NSUB = KP == 64 ? ZGR_N64 : (KP == 32 ? ZGR_N32 : ZGR_N16);   // adjacent tiles per row block that share one U tile
  static constexpr int STAGES = KP == 64 ? ZGR_S64 : (KP == 32 ? ZGR_S32 : ZGR_S16);  // theta tiles in flight (loaded, transformed in place, stored)
  static constexpr int USTAGES = 2;                        // U tiles in flight
  static constexpr int NACC = WIDE ? 2 : 4;                // accumulator buffers in tensor memory
  static constexpr int ROWB = KP * 2;                      // bytes per row of the U and G operands
  static constexpr int THETA_BYTES = 128 * NS * 2;         // NS/64 boxes of 128 rows x 128 B
  static constexpr int U_BYTES = 128 * ROWB;               // one of hi / lo
  static constexpr int G_BYTES = NS * ROWB;                // one of hi / lo, one tile's strip
  static constexpr int ID_BYTES = 1024;                    // 16 x 16 identity (512 B), padded to the swizzle alignment
  static constexpr int BAR_BYTES = 1024;
  static constexpr int SMEM_BYTES =
      STAGES * THETA_BYTES + USTAGES * 2 * U_BYTES + NSUB * 2 * G_BYTES + ID_BYTES + BAR_BYTES + 1024 /* alignment slack */;
  static constexpr int TMEM_COLS = NACC * NS <= 256 ? 256 : 512;   // allocations are powers of two
  static_assert(SMEM_BYTES <= 232448, "shared-memory budget of one CTA");
};

struct TileCoord {
  int32_t tensor;
  int32_t col0;
  int32_t row0;
  int32_t ncols;   // columns of this tile that exist in the tensor (<= 128)
};

}  // namespace

// Work item = NSUB adjacent column tiles (a strip of up to 128*NSUB columns) x a range of rows.
// Tiles are visited row block by row block, the NSUB tiles of a row block one after the other, so
// that a CTA touches up to 256*NSUB contiguous bytes of every row and loads each U tile once.
// STATS = true turns the same pipeline into the norm bookkeeping: no weights are loaded or stored,
// D = b U G only, and the epilogue accumulates sum (a Z)^2, sum (b U G)^2 and sum z^2 per tensor
// (term[0].iso carries the scale a, term[0].cb = b; the sums go to the work item's bookkeeping slots).
// MULTI = true applies several (seed, coefficient) terms in the one pass: the coefficient strips of
// the terms are summed before the split (U (sum_q c_q b G_q) is one product), the isotropic normals
// are added term by term in the epilogue.
// ZOUT = true is the test hook of this kernel: the same loads, products and epilogue arithmetic, but the fp32
// result of every element (accumulator plus normals, before the rounding to the storage type) goes to
// p.zout[row * cols + col] by plain stores and nothing is written back to the weights.  On a zeroed
// weight image with coefficient 1 that is z itself as this kernel computes it.
// SSTATS = true (single-term sweeps) is the sweep itself with the norm bookkeeping folded in: before a thread
// overwrites its 16 bytes of the staged tile it reads theta back from them, so that the guided part (accumulator
// minus theta) and the whole step (result minus theta) can be squared and summed; the isotropic part costs one
// addition per pair of normals (the squared radius is the argument of the square root).  The sums are of
// (c a Z)^2, (c b U G)^2 and (c z)^2; the host divides by c^2.
template <typename T, int BITS, int KP, bool STATS = false, bool MULTI = false, bool ZOUT = false, bool SSTATS = false>
__global__ void __launch_bounds__(UmmaCfg<KP>::THREADS, 1) sweep_umma_kernel(const __grid_constant__ SweepParams p, const CUtensorMap* __restrict__ tmaps,
                                                                     int* __restrict__ error) {
  using Cfg = UmmaCfg<KP>;
  constexpr int NS = Cfg::NS, S = Cfg::STAGES, US = Cfg::USTAGES, ROWB = Cfg::ROWB, NACC = Cfg::NACC, NSUB = Cfg::NSUB;
  constexpr int kEpiWarps = Cfg::EPI_WARPS, kUmmaThreads = Cfg::THREADS;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint8_t* theta_base = smem;                                           // S tiles
  uint8_t* u_base = theta_base + S * Cfg::THETA_BYTES;                  // US x (hi, lo)
  uint8_t* g_base = u_base + US * 2 * Cfg::U_BYTES;                     // NSUB x (hi, lo)
  uint8_t* ident = g_base + NSUB * 2 * Cfg::G_BYTES;
  uint64_t* bars = reinterpret_cast<uint64_t*>(ident + Cfg::ID_BYTES);
  const uint32_t bar0 = smem_u32(bars);
  auto BAR_FULL = [&](int s) { return bar0 + 8u * static_cast<uint32_t>(s); };                          // theta tile landed
  auto BAR_OUT = [&](int s) { return bar0 + 8u * static_cast<uint32_t>(S + s); };                       // result written into the stage
  auto BAR_ACC_FULL = [&](int b) { return bar0 + 8u * static_cast<uint32_t>(2 * S + b); };              // accumulator complete
  auto BAR_ACC_EMPTY = [&](int b) { return bar0 + 8u * static_cast<uint32_t>(2 * S + NACC + b); };      // accumulator read out
  auto BAR_U_FULL = [&](int u) { return bar0 + 8u * static_cast<uint32_t>(2 * S + 2 * NACC + u); };     // U tile landed
  auto BAR_U_FREE = [&](int u) { return bar0 + 8u * static_cast<uint32_t>(2 * S + 2 * NACC + US + u); };  // U tile consumed
  const uint32_t BAR_G = bar0 + 8u * static_cast<uint32_t>(2 * S + 2 * NACC + 2 * US);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * S + 2 * NACC + 2 * US + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    constexpr int kWarpsPerTile = kEpiWarps / Cfg::GROUPS;   // epilogue warps that work on one tile
    for (int s = 0; s < S; ++s) {
      mbar_init(BAR_FULL(s), 1);
      mbar_init(BAR_OUT(s), kWarpsPerTile);
    }
    for (int b = 0; b < NACC; ++b) {
      mbar_init(BAR_ACC_FULL(b), 1);
      mbar_init(BAR_ACC_EMPTY(b), kWarpsPerTile);
    }
    for (int u = 0; u < US; ++u) {
      mbar_init(BAR_U_FULL(u), 1);
      mbar_init(BAR_U_FREE(u), 1);
    }
    mbar_init(BAR_G, kEpiWarps);
    *abort_flag = 0;
    fence_mbar_init();
  }
  // 16 x 16 identity in the storage type, K-major rows of 32 bytes, 32-byte swizzle
  for (int i = threadIdx.x; i < 256; i += kUmmaThreads) {
    const int n = i >> 4, k = i & 15;
    *reinterpret_cast<uint16_t*>(ident + swizzle(static_cast<uint32_t>(n * 32 + k * 2), 32)) = (n == k) ? Pack16<T>::kOne : uint16_t(0);
  }
  fence_proxy_async();
  __syncthreads();
  if (warp == 1) {
    tmem_alloc(smem_u32(tmem_slot), Cfg::TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  if (warp < 2) dependency_begin(p);      // (the epilogue warps: after the first strip, which is made of the seed alone)
  // this CTA's items: a contiguous share, or every gridDim.x-th one
  const int it_first = p.starts ? p.starts[blockIdx.x] : static_cast<int>(blockIdx.x);
  const int it_end = p.starts ? p.starts[blockIdx.x + 1] : p.n_items, it_step = p.starts ? 1 : static_cast<int>(gridDim.x);

  // The three roles walk the same sequence of (item, row block, tile) triples; t counts tiles and
  // rb counts row blocks over the whole life of the CTA, which fixes every ring slot and phase.
  if (warp == 0) {
    // ===================================== TMA producer =====================================
    if (elect_one()) {
      TileCoord ring[S];
      int t = 0, rb = 0;
      bool ok = true;
      auto store_tile = [&](int s) {
        const TileCoord& o = ring[s];
        const CUtensorMap* tm = tmaps + 3 * o.tensor;
        const uint32_t src = smem_u32(theta_base + s * Cfg::THETA_BYTES);
        for (int c = 0; c * 64 < o.ncols; ++c) tma_store_2d(tm, o.col0 + 64 * c, o.row0, src + c * 16384);
        tma_commit();
      };
      for (int it = it_first; it < it_end && ok; it += it_step) {
        const WorkItem w = p.items[it];
        const CUtensorMap* tm = tmaps + 3 * w.tensor;
        const int row_end = static_cast<int>(w.row0_or_e0 + w.nrows_or_count);
        const int nsub = (w.ncols + NS - 1) / NS;
        for (int row0 = static_cast<int>(w.row0_or_e0); row0 < row_end && ok; row0 += 128, ++rb) {
          const int u = rb % US;
          if (rb >= US && !mbar_wait<true>(BAR_U_FREE(u), ((rb / US) - 1) & 1, abort_flag, error, 8)) { ok = false; break; }
          const uint32_t udst = smem_u32(u_base + u * 2 * Cfg::U_BYTES);
          mbar_arrive_expect_tx(BAR_U_FULL(u), static_cast<uint32_t>(2 * Cfg::U_BYTES));
          tma_load_2d(udst, tm + 1, 0, row0, BAR_U_FULL(u));
          tma_load_2d(udst + Cfg::U_BYTES, tm + 2, 0, row0, BAR_U_FULL(u));
          for (int sub = 0; sub < nsub && !STATS; ++sub, ++t) {
            const int s = t % S;
            if (t >= S) {
              // the epilogue has written tile t-S into this stage: store it, then the stage is free
              if (!mbar_wait<true>(BAR_OUT(s), ((t / S) - 1) & 1, abort_flag, error, 1)) { ok = false; break; }
              if (!ZOUT) {
                store_tile(s);
                tma_wait_read0();
              }
            }
            const int col0 = static_cast<int>(w.col0) + NS * sub;
            const int ncols = min(NS, w.ncols - NS * sub);
            ring[s] = TileCoord{w.tensor, col0, row0, ncols};
            const int nbox = (ncols + 63) / 64;
            const uint32_t dst = smem_u32(theta_base + s * Cfg::THETA_BYTES);
            mbar_arrive_expect_tx(BAR_FULL(s), static_cast<uint32_t>(nbox * 16384));
            for (int c = 0; c < nbox; ++c) tma_load_2d(dst + c * 16384, tm, col0 + 64 * c, row0, BAR_FULL(s));
          }
        }
      }
      // drain: store the last tiles
      const int total = t;
      for (int v = (total > S ? total - S : 0); v < total && ok && !STATS; ++v) {
        if (!mbar_wait<true>(BAR_OUT(v % S), (v / S) & 1, abort_flag, error, 2)) { ok = false; break; }
        if (!ZOUT) store_tile(v % S);
      }
      if (!ok) {
        // aborting: let the loads already issued land before the CTA gives up its shared memory
        for (int v = (total > S ? total - S : 0); v < total; ++v) {
          const unsigned long long t0 = clock64();
          while (!mbar_try_wait(BAR_FULL(v % S), (v / S) & 1) && clock64() - t0 < kWaitLimitCycles) {
          }
        }
        for (int v = (rb > US ? rb - US : 0); v < rb; ++v) {
          const unsigned long long t0 = clock64();
          while (!mbar_try_wait(BAR_U_FULL(v % US), (v / US) & 1) && clock64() - t0 < kWaitLimitCycles) {
          }
        }
      }
      tma_wait_all0();
    }
  } else if (warp == 1) {
    // ===================================== MMA issuer =====================================
    if (elect_one()) {
      const uint32_t idesc_id = make_idesc(Pack16<T>::kFmt, 16);
      const uint32_t idesc_ug = make_idesc(0, NS);          // fp16 operands
      const uint64_t desc_id = make_desc(smem_u32(ident), 32);
      // Descriptors differ only in their start-address field (bits 0-13, address >> 4), so every
      // operand below is one of these bases plus a small constant.
      const uint64_t desc_theta0 = make_desc(smem_u32(theta_base), 128);
      const uint64_t desc_u0 = make_desc(smem_u32(u_base), ROWB);
      const uint64_t desc_g0 = make_desc(smem_u32(g_base), ROWB);
      int t = 0, rb = 0, item_no = 0;
      bool ok = true;
      for (int it = it_first; it < it_end && ok; it += it_step, ++item_no) {
        const WorkItem w = p.items[it];
        const int sh = acc_shift(p.tensors[w.tensor], p);
        if (!mbar_wait<true>(BAR_G, item_no & 1, abort_flag, error, 3)) break;
        tc_fence_after();
        const int row_end = static_cast<int>(w.row0_or_e0 + w.nrows_or_count);
        const int nsub = (w.ncols + NS - 1) / NS;
        for (int row0 = static_cast<int>(w.row0_or_e0); row0 < row_end && ok; row0 += 128, ++rb) {
          const int u = rb % US;
          if (!mbar_wait<true>(BAR_U_FULL(u), (rb / US) & 1, abort_flag, error, 9)) { ok = false; break; }
          const uint64_t desc_uhi = desc_u0 + static_cast<uint64_t>((u * 2 * Cfg::U_BYTES) >> 4);
          const uint64_t desc_ulo = desc_uhi + static_cast<uint64_t>(Cfg::U_BYTES >> 4);
          for (int sub = 0; sub < nsub; ++sub, ++t) {
            const int s = t % S, b = t % NACC;
            if (t >= NACC && !mbar_wait<true>(BAR_ACC_EMPTY(b), ((t / NACC) - 1) & 1, abort_flag, error, 5)) { ok = false; break; }
            tc_fence_after();
            const uint64_t desc_theta = desc_theta0 + static_cast<uint64_t>((s * Cfg::THETA_BYTES) >> 4);
            const uint32_t d = tmem_base + static_cast<uint32_t>(b * NS);
            const int nbox = (min(NS, w.ncols - NS * sub) + 63) / 64;
            // 2^s c b U G, split operands
            const uint64_t desc_ghi = desc_g0 + static_cast<uint64_t>((sub * 2 * Cfg::G_BYTES) >> 4);
            const uint64_t desc_glo = desc_ghi + static_cast<uint64_t>(Cfg::G_BYTES >> 4);
#pragma unroll
            for (int k = 0; k < KP / 16; ++k)
              umma(d, desc_ulo + static_cast<uint64_t>(2 * k), desc_ghi + static_cast<uint64_t>(2 * k), idesc_ug, k == 0 ? 0u : 1u);
#pragma unroll
            for (int k = 0; k < KP / 16; ++k) umma(d, desc_uhi + static_cast<uint64_t>(2 * k), desc_glo + static_cast<uint64_t>(2 * k), idesc_ug, 1u);
#pragma unroll
            for (int k = 0; k < KP / 16; ++k) umma(d, desc_uhi + static_cast<uint64_t>(2 * k), desc_ghi + static_cast<uint64_t>(2 * k), idesc_ug, 1u);
            // theta last, 16 columns at a time:  D <- theta I + 2^-s D
            if (!STATS) {
              if (!mbar_wait<true>(BAR_FULL(s), (t / S) & 1, abort_flag, error, 4)) { ok = false; break; }
              tc_fence_after();
#define ZGR_THETA_IN(SC)                                                                                                   \
  _Pragma("unroll") for (int c = 0; c < NS / 64; ++c) {                                                                    \
    if (c < nbox) {                                                                                                        \
      _Pragma("unroll") for (int k = 0; k < 4; ++k)                                                                        \
          umma_scaled_d<SC>(d + static_cast<uint32_t>(64 * c + 16 * k), desc_theta + static_cast<uint64_t>((c * 16384 + 32 * k) >> 4), \
                            desc_id, idesc_id);                                                                            \
    }                                                                                                                      \
  }
              switch (sh) {
                case 0: ZGR_THETA_IN(0) break;
                case 1: ZGR_THETA_IN(1) break;
                case 2: ZGR_THETA_IN(2) break;
                case 3: ZGR_THETA_IN(3) break;
                case 4: ZGR_THETA_IN(4) break;
                case 5: ZGR_THETA_IN(5) break;
                case 6: ZGR_THETA_IN(6) break;
                case 7: ZGR_THETA_IN(7) break;
                case 8: ZGR_THETA_IN(8) break;
                case 9: ZGR_THETA_IN(9) break;
                case 10: ZGR_THETA_IN(10) break;
                case 11: ZGR_THETA_IN(11) break;
                case 12: ZGR_THETA_IN(12) break;
                case 13: ZGR_THETA_IN(13) break;
                case 14: ZGR_THETA_IN(14) break;
                default: ZGR_THETA_IN(15) break;
              }
#undef ZGR_THETA_IN
            }
            umma_commit(BAR_ACC_FULL(b));
          }
          if (ok) umma_commit(BAR_U_FREE(u));   // arrives once every product that reads this U tile has completed
        }
      }
    }
  } else {
    // ===================================== epilogue warps =====================================
    // Warp (quad, cgrp) owns rows 32 quad .. 32 quad + 31 and columns 32 cgrp .. 32 cgrp + 31 of every tile.
    const int e = warp - 2;                 // 0..15
    const int quad = warp & 3;              // tensor-memory lane quadrant this warp may read
    constexpr int GROUPS = Cfg::GROUPS;                                      // each warp covers GROUPS column groups of its tiles
    const int grp = e / (kEpiWarps / GROUPS);                                // which tiles: t % GROUPS == grp
    const int cg_first = ((e >> 2) % (kEpiWarps / 4 / GROUPS)) * GROUPS;     // first 32-column group of this warp
    const int et = e * 32 + lane;
    const uint32_t tmem_row = tmem_base + (static_cast<uint32_t>(32 * quad) << 16);
    const int row_in_tile = 32 * quad + lane;
    const uint32_t row_xor16 = static_cast<uint32_t>(row_in_tile & 7) << 4;   // 128-byte swizzle: the 16-byte chunk index is xor-ed with the row
    const uint32_t theta_s32 = smem_u32(theta_base);
    const uint32_t g_s32 = smem_u32(g_base);
    int t = 0, item_no = 0;
    bool ok = true;
    for (int it = it_first; it < it_end && ok; it += it_step, ++item_no) {
      const WorkItem w = p.items[it];
      const TensorDesc& td = p.tensors[w.tensor];
      const uint32_t tid = static_cast<uint32_t>(td.id);
      const int r = td.rank;
      const uint64_t tcols = static_cast<uint64_t>(td.cols);   // kept in a register: the barriers below force reloads of anything read through td
      const int sh = acc_shift(td, p);
      const PhiloxPre pre = philox_pre(0u, tid, p.term[0].keys);
      const float gscale = __int_as_float((127 + sh - td.ushift) << 23);   // 2^(s - j): the strips hold c b G 2^(s - j)
      if (GROUPS > 1 && t > 0) {
        // The strips are about to be overwritten.  With two groups this warp may be one tile ahead of the
        // other group, whose last tile of the previous item can still have products in flight that read the
        // old strips: wait until that tile's accumulator is complete (no later product exists before BAR_G).
        const int tp = t - 1;
        if (!mbar_wait<false>(BAR_ACC_FULL(tp % NACC), (tp / NACC) & 1, abort_flag, error, 11)) break;
      }
      // (codes that earlier work in the stream delivers may only be read behind it)
      if (item_no == 0 && td.q != nullptr) dependency_begin(p);
      // ---- coefficient strips c b G -> K-major hi/lo operands, one per tile of a row block ----
      for (int idx = et; idx < (KP / 2) * (NSUB * NS / 8); idx += kEpiWarps * 32) {
        // consecutive lanes take consecutive pairs of rows k of the same columns: their 32-bit stores below then
        // fall into KP/2 consecutive words of one operand row (with the octet index fastest they would all hit
        // one bank: 27 wavefronts per store instead of 2)
        const int kp = idx % (KP / 2), o = idx / (KP / 2);
        const int cc = 8 * o;                       // column within the item's strip
        if (cc >= ((w.ncols + NS - 1) / NS) * NS) continue;   // tiles of this item that do not exist
        float g0[8], g1[8];
        if (cc < w.ncols && 2 * kp < r) {
          guided8<BITS, false, MULTI>(td, p, 2 * kp, w.col0 + cc, g0);
        } else {
#pragma unroll
          for (int i = 0; i < 8; ++i) g0[i] = 0.0f;
        }
        if (cc < w.ncols && 2 * kp + 1 < r) {
          guided8<BITS, false, MULTI>(td, p, 2 * kp + 1, w.col0 + cc, g1);
        } else {
#pragma unroll
          for (int i = 0; i < 8; ++i) g1[i] = 0.0f;
        }
        const uint32_t g_hi = g_s32 + static_cast<uint32_t>((cc / NS) * 2 * Cfg::G_BYTES);
        const uint32_t g_lo = g_hi + static_cast<uint32_t>(Cfg::G_BYTES);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          uint32_t hi, lo;
          split_f16(g0[i] * gscale, g1[i] * gscale, hi, lo);
          const uint32_t off = swizzle(static_cast<uint32_t>(((cc % NS) + i) * ROWB + 4 * kp), ROWB);
          sts32(g_hi + off, hi);
          sts32(g_lo + off, lo);
        }
      }
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(BAR_G);
      if (item_no == 0 && td.q == nullptr) dependency_begin(p);
      // The epilogue warps of a scheduler run the same instruction stream from the same starting
      // point: first the integer rounds of the generator, then the special-function half of the
      // transform.  Holding every other column group back once per item puts half of each scheduler's
      // warps in the other phase, so the two pipes overlap (measured with one group: 6.5 -> 6.15 ms per 7B sweep;
      // with two groups the groups are out of step by construction).
      if (GROUPS == 1 && (cg_first & 1)) __nanosleep(kStaggerNs);

      const int row_end = static_cast<int>(w.row0_or_e0 + w.nrows_or_count);
      const int nsub = (w.ncols + NS - 1) / NS;
      double sum_iso = 0.0, sum_gd = 0.0, sum_z = 0.0;   // STATS / SSTATS only
      for (int row0 = static_cast<int>(w.row0_or_e0); row0 < row_end && ok; row0 += 128) {
        const int64_t row = static_cast<int64_t>(row0) + row_in_tile;
        const uint64_t row_oct0 = (static_cast<uint64_t>(row) * tcols + static_cast<uint64_t>(w.col0)) >> 3;   // octet index of the strip's first column in this row
        for (int sub = 0; sub < nsub; ++sub, ++t) {
          if (GROUPS > 1 && (t % GROUPS) != grp) continue;     // another group's tile
          const int s = t % S, b = t % NACC;
          if (!mbar_wait<false>(BAR_ACC_FULL(b), (t / NACC) & 1, abort_flag, error, 6)) { ok = false; break; }
          tc_fence_after();
#pragma unroll
          for (int pass = 0; pass < GROUPS; ++pass) {
          const int cgrp = cg_first + pass;                // which 32 columns of the tile
          const uint32_t tmem_warp = tmem_row + static_cast<uint32_t>(32 * cgrp);
          const uint32_t chunk0 = static_cast<uint32_t>(((32 * cgrp) & 63) >> 3);
          const uint32_t out_off = static_cast<uint32_t>(((32 * cgrp) >> 6) * 16384 + row_in_tile * 128);
          if (NS * sub + 32 * cgrp < w.ncols) {
            const uint64_t oct0 = row_oct0 + static_cast<uint64_t>((NS * sub + 32 * cgrp) >> 3);
            const uint32_t oct0_lo = static_cast<uint32_t>(oct0);     // (the planner keeps tensors of 2^34 elements and more away from here)
            // the row's 128 bytes in the staged tile start on a 128-byte boundary, so the swizzled chunk offset
            // (bits 4..6) can be xor-ed in rather than added: one logic instruction per chunk
            const uint32_t out_box = (theta_s32 + static_cast<uint32_t>(s * Cfg::THETA_BYTES) + out_off) ^ row_xor16;
            uint32_t h0[16], h1[16];
            tmem_ld16(tmem_warp + static_cast<uint32_t>(b * NS), h0);
            tmem_ld16(tmem_warp + static_cast<uint32_t>(b * NS + 16), h1);
            tmem_ld_wait();
            if constexpr (STATS) {
              const float descale = __int_as_float((127 - sh) << 23);
              float f_iso = 0.0f, f_gd = 0.0f, f_z = 0.0f;
#pragma unroll
              for (int o = 0; o < 4; ++o) {
                float zi[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) zi[i] = 0.0f;
                normals8_acc_pre<BITS>(p.term[0].keys, pre, oct0_lo + static_cast<uint32_t>(o), p.term[0].iso, zi);
                const bool live = row < row_end && NS * sub + 32 * cgrp + 8 * o < w.ncols;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                  const float gd = __uint_as_float(o < 2 ? h0[8 * (o & 1) + i] : h1[8 * (o & 1) + i]) * descale;   // no identity product here: undo 2^s
                  if (live) {
                    f_iso = fmaf(zi[i], zi[i], f_iso);
                    f_gd = fmaf(gd, gd, f_gd);
                    f_z = fmaf(zi[i] + gd, zi[i] + gd, f_z);
                  }
                }
              }
              sum_iso += static_cast<double>(f_iso);
              sum_gd += static_cast<double>(f_gd);
              sum_z += static_cast<double>(f_z);
            } else {
            if constexpr (SSTATS) {
#pragma unroll
              for (int o = 0; o < 4; ++o) {
                float acc[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) acc[i] = __uint_as_float(o < 2 ? h0[8 * (o & 1) + i] : h1[8 * (o & 1) + i]);
                const uint32_t chunk_addr = out_box ^ ((chunk0 + static_cast<uint32_t>(o)) << 4);
                float th[8];
                unpack8<T>(lds128(chunk_addr), th);                      // theta, before this thread overwrites it
                float f_iso = 0.0f, f_gd = 0.0f, f_z = 0.0f;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                  const float gd = acc[i] - th[i];
                  f_gd = fmaf(gd, gd, f_gd);
                }
                normals8_acc_pre_rsum<BITS, true>(p.term[0].keys, pre, oct0_lo + static_cast<uint32_t>(o), p.term[0].iso, acc, f_iso);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                  const float zc = acc[i] - th[i];
                  f_z = fmaf(zc, zc, f_z);
                }
                if (row < row_end && NS * sub + 32 * cgrp + 8 * o < w.ncols) {
                  sum_iso += static_cast<double>(f_iso);
                  sum_gd += static_cast<double>(f_gd);
                  sum_z += static_cast<double>(f_z);
                }
                sts128(chunk_addr, make_uint4(Pack16<T>::pack(acc[0], acc[1]), Pack16<T>::pack(acc[2], acc[3]), Pack16<T>::pack(acc[4], acc[5]),
                                              Pack16<T>::pack(acc[6], acc[7])));
              }
            } else {
              // four octets per thread, one generator chain after the other, each beside the transform of the octet before it (see
              // normals8_acc_linked; with 32 random bits per normal, where an octet is two generator blocks, only the order of the
              // octets is kept: 3615 -> 3540 us on four LLaMA-7B-shaped layers)
              float acc[4][8];
              const uint32_t zero = static_cast<uint32_t>(p.early) >> 1;      // (early is 0 or 1)
              uint32_t link = 0;
#pragma unroll
              for (int o = 0; o < 4; ++o)
#pragma unroll
                for (int i = 0; i < 8; ++i) acc[o][i] = __uint_as_float(o < 2 ? h0[8 * (o & 1) + i] : h1[8 * (o & 1) + i]);
#pragma unroll
              for (int o = 0; o < 4; ++o) {
                if constexpr (BITS == 32) {
                  normals8_acc_pre<BITS>(p.term[0].keys, pre, oct0_lo + static_cast<uint32_t>(o), p.term[0].iso, acc[o]);
                  asm volatile("" ::: "memory");
                } else {
                  normals8_acc_linked(p.term[0].keys, pre, oct0_lo + static_cast<uint32_t>(o), p.term[0].iso, zero, link, acc[o]);
                }
              }
              if (MULTI) {
                // term by term over all four octets: the keys are fetched once per term
#pragma unroll 1
                for (int q = 1; q < p.n_terms; ++q) {
                  const PhiloxKeys& keys = p.term[q].keys;
                  const PhiloxPre pre_q = philox_pre(0u, tid, keys);
#pragma unroll
                  for (int o = 0; o < 4; ++o) {
                    if constexpr (BITS == 32) normals8_acc_pre<BITS>(keys, pre_q, oct0_lo + static_cast<uint32_t>(o), p.term[q].iso, acc[o]);
                    else normals8_acc_linked(keys, pre_q, oct0_lo + static_cast<uint32_t>(o), p.term[q].iso, zero, link, acc[o]);
                  }
                }
              }
#pragma unroll
            for (int o = 0; o < 4; ++o) {
              if constexpr (ZOUT) {
                const int col = NS * sub + 32 * cgrp + 8 * o;          // within the item's strip
                if (row < row_end && col < w.ncols) {
                  float4* dst = reinterpret_cast<float4*>(p.zout + static_cast<uint64_t>(row) * tcols + static_cast<uint64_t>(w.col0 + col));
                  dst[0] = make_float4(acc[o][0], acc[o][1], acc[o][2], acc[o][3]);
                  dst[1] = make_float4(acc[o][4], acc[o][5], acc[o][6], acc[o][7]);
                }
              } else {
                const uint4 q = make_uint4(Pack16<T>::pack(acc[o][0], acc[o][1]), Pack16<T>::pack(acc[o][2], acc[o][3]),
                                           Pack16<T>::pack(acc[o][4], acc[o][5]), Pack16<T>::pack(acc[o][6], acc[o][7]));
                sts128(out_box ^ ((chunk0 + static_cast<uint32_t>(o)) << 4), q);
              }
            }
            }
            }
          }
          }
          tc_fence_before();
          fence_proxy_async();
          __syncwarp();
          if (lane == 0) {
            mbar_arrive(BAR_ACC_EMPTY(b));
            if (!STATS) mbar_arrive(BAR_OUT(s));
          }
        }
      }
      if constexpr (STATS || SSTATS) {
        if (ok) store_item_stats(p, it, e, sum_iso, sum_gd, sum_z);   // one slot per epilogue warp (at most kStatSlots of them)
      }
    }
  }

  // ---- common exit ----
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, Cfg::TMEM_COLS);
  }
}

size_t umma_smem_bytes(int kpad) {
  return kpad == 16 ? UmmaCfg<16>::SMEM_BYTES : (kpad == 32 ? UmmaCfg<32>::SMEM_BYTES : UmmaCfg<64>::SMEM_BYTES);
}
int umma_strip_cols(int kpad) { return kpad == 64 ? UmmaCfg<64>::NS * UmmaCfg<64>::NSUB : (kpad == 32 ? UmmaCfg<32>::NS * UmmaCfg<32>::NSUB : UmmaCfg<16>::NS * UmmaCfg<16>::NSUB); }

namespace {
template <typename T, int BITS, bool STATS = false, bool MULTI = false, bool ZOUT = false, bool SSTATS = false>
cudaError_t launch_umma_kp(int kpad, const SweepParams& p, const CUtensorMap* tmaps, int* error, int grid, cudaStream_t st) {
  static_assert(UmmaCfg<16>::EPI_WARPS <= kStatSlots && UmmaCfg<32>::EPI_WARPS <= kStatSlots && UmmaCfg<64>::EPI_WARPS <= kStatSlots,
                "one bookkeeping slot per epilogue warp");
#define ZGR_LAUNCH_UMMA(KPV)                                                                                       \
  {                                                                                                                \
    auto k = sweep_umma_kernel<T, BITS, KPV, STATS, MULTI, ZOUT, SSTATS>;                                                 \
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, UmmaCfg<KPV>::SMEM_BYTES); \
    if (e != cudaSuccess) return e;                                                                                \
    return launch_sweep_kernel(k, grid, UmmaCfg<KPV>::THREADS, UmmaCfg<KPV>::SMEM_BYTES, st, p, tmaps, error);                \
  }
  if (kpad == 16) ZGR_LAUNCH_UMMA(16)
  else if (kpad == 32) ZGR_LAUNCH_UMMA(32)
  else ZGR_LAUNCH_UMMA(64)
#undef ZGR_LAUNCH_UMMA
}
}  // namespace

namespace {
template <typename T>
cudaError_t launch_umma_typed(const KernelChoice& kc, const SweepParams& p, const CUtensorMap* tmaps, int* error, int grid, cudaStream_t st) {
  if (p.n_terms > 1) {
    return kc.bits == 32 ? launch_umma_kp<T, 32, false, true>(kc.kpad, p, tmaps, error, grid, st)
                         : launch_umma_kp<T, 16, false, true>(kc.kpad, p, tmaps, error, grid, st);
  }
  if (p.item_stats != nullptr) {   // the sweep also accumulates the norm bookkeeping
    return kc.bits == 32 ? launch_umma_kp<T, 32, false, false, false, true>(kc.kpad, p, tmaps, error, grid, st)
                         : launch_umma_kp<T, 16, false, false, false, true>(kc.kpad, p, tmaps, error, grid, st);
  }
  return kc.bits == 32 ? launch_umma_kp<T, 32>(kc.kpad, p, tmaps, error, grid, st) : launch_umma_kp<T, 16>(kc.kpad, p, tmaps, error, grid, st);
}
}  // namespace

cudaError_t launch_sweep_umma(const KernelChoice& kc, const SweepParams& p, const CUtensorMap* tmaps, int* error, int grid, cudaStream_t st) {
  if (kc.dtype == 2) return launch_umma_typed<__nv_bfloat16>(kc, p, tmaps, error, grid, st);
  if (kc.dtype == 1) return launch_umma_typed<__half>(kc, p, tmaps, error, grid, st);
  return cudaErrorInvalidValue;
}

cudaError_t launch_debug_z_umma(const KernelChoice& kc, const SweepParams& p, const CUtensorMap* tmaps, int* error, int grid, cudaStream_t st) {
  if (p.zout == nullptr || p.n_terms != 1) return cudaErrorInvalidValue;
  if (kc.dtype == 2)
    return kc.bits == 32 ? launch_umma_kp<__nv_bfloat16, 32, false, false, true>(kc.kpad, p, tmaps, error, grid, st)
                         : launch_umma_kp<__nv_bfloat16, 16, false, false, true>(kc.kpad, p, tmaps, error, grid, st);
  if (kc.dtype == 1)
    return kc.bits == 32 ? launch_umma_kp<__half, 32, false, false, true>(kc.kpad, p, tmaps, error, grid, st)
                         : launch_umma_kp<__half, 16, false, false, true>(kc.kpad, p, tmaps, error, grid, st);
  return cudaErrorInvalidValue;
}

cudaError_t launch_stats_umma(const KernelChoice& kc, const SweepParams& p, const CUtensorMap* tmaps, int* error, int grid, cudaStream_t st) {
  // the storage type plays no role when no weights are touched: one instantiation serves all
  return kc.bits == 32 ? launch_umma_kp<__nv_bfloat16, 32, true>(kc.kpad, p, tmaps, error, grid, st)
                       : launch_umma_kp<__nv_bfloat16, 16, true>(kc.kpad, p, tmaps, error, grid, st);
}

}  // namespace zgr
