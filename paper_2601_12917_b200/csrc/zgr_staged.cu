// Sweep with a three-part tensor-core contraction and weights staged by TMA, for guided tensors that zgr_umma.cu does not take: fp32
// storage, 16-bit rows that are no multiple of eight elements long, and sets of rank <= 8 that are worth a tensor-core
// kernel (tensor_core_kind and staged_kind in zgr_host.cu have the sizes).
//     theta <- rnd(theta + c (a Z + b U G))            (Eq. (perturbation) applied as in Algorithm 1)
//
// Rows of any length.  Generator blocks run along the flattened tensor, eight elements ("an octet") at a time, so where the row
// length is no multiple of eight the octets of row m start at column  h_m = -(m cols) mod 8,  and TMA, which wants 16-byte
// boundaries and pitches, cannot address the rows.  Both depend on m mod 8 alone: the rows m = i (mod 8) form a matrix of pitch
// 8 cols whose whole octets start at element i cols + h_i, a multiple of eight.  Such a tensor therefore has eight tensor maps, one
// per residue i, each as wide as the whole octets of its rows.  A tile of 128 rows takes 32 rows of each of four residues, one per quarter
// of the tensor memory, so that everything within a warp has the same shift, which goes into the column of its tensor-memory
// load.  Two tiles (residues 0-3 and 4-7) cover 256 consecutive rows; the library's copy of U keeps its rows in that order
// (staged_copy_row), so that U stays one contiguous tile.  What is left of a row, the columns before its first and behind its last whole
// octet, is done element by element by the warps that own the ends (finish_part).  In tensors of whole octets a tile is 128
// consecutive rows and nothing is left over.
//
// Pipeline (one CTA per SM; small sets give it a contiguous share of the items, otherwise its first item is its own index and
// the others come from a counter in global memory):
//   warp 0   hands out the items through a ring of four; TMA loads of U (128 rows, three bf16 parts) and of the weights, and
//            the TMA stores of finished tiles, a lane per box
//   warp 1   tcgen05.mma:  D = c b U G  (fp32, six products of bf16 parts) into a ring of tensor-memory buffers
//   warps 2-17  coefficient strips c b G into shared memory, one item ahead where two strips fit; then, in two groups on
//            alternate tiles, 32 rows x 128 bytes per warp, a thread per row: D from tensor memory, the normals, the weights from
//            the staged tile and the result back into it
// A tile is 128 rows x 256 bytes: 128 columns of 16-bit weights, 64 of fp32 (two such tiles share a strip and a tile of U).
//
// Against sweep_tile_kernel, which loads the weights from global memory an octet per thread and turns the products round through
// shared memory, the address arithmetic, the transposition and the exposed loads are gone.
//
// Operand precision.  An fp32 number is the sum of three bf16 numbers (8 bits each) without error, up to the largest bf16 number in size
// (3.39e38; beyond it, and for infinities, the parts that follow the first are not numbers, and neither is what they are multiplied into);
// six of the nine products are formed, the others are below 2^-24 of the result.  With the copies of U leaning against
// the truncation of the tensor cores (truncation_lean) the contraction is as accurate as a chain of fp32 multiply-adds, from
// rank 2 on more so.  The perturbation is summed on its own scale and added to the weight once.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <type_traits>

#include "zgr_device.cuh"
#include "zgr_kernels.h"
#include "zgr_strip.cuh"
#include "zgr_tcgen05.cuh"

namespace zgr {
namespace {

constexpr int kThreadsStaged = 32 * (2 + kEpi);
constexpr int kGroupWarps = kEpi / 2;          // epilogue warps that work on one tile
constexpr int kRing = 4;                       // items published ahead
constexpr int kTileBytes = 128 * 256;
constexpr int kBoxBytes = 32 * 128;            // 32 rows x 128 bytes
constexpr int kMaxStages = 5;
constexpr int kTmemBase = 16;                  // (the head of a row is read from up to seven columns before its buffer)

template <typename T>
struct StagedCfg {
  static constexpr int COLS = 256 / static_cast<int>(sizeof(T));     // columns per tile
  static constexpr int HALF = COLS / 2;                              // columns per warp
  static constexpr int NSUB = 128 / COLS;                            // tiles of a row block
  static constexpr int ACC_COLS = COLS + 16;                         // tensor-memory columns per buffer
  static constexpr int NACC = sizeof(T) == 4 ? 4 : 3;
};

// Shared-memory plan for contraction width kp (16, 32, 64).
struct StagedSmem {
  int rowb, u_bytes, g_bytes, u_stages, g_stages, stages, total;
};
__host__ __device__ inline StagedSmem staged_smem(int kp) {
  StagedSmem s;
  s.rowb = 2 * kp;
  s.u_bytes = 128 * s.rowb;
  s.g_bytes = kTileN * s.rowb;
  s.u_stages = kp == 16 ? 2 : 1;
  s.g_stages = kp == 64 ? 1 : 2;
  s.stages = kp == 16 ? 5 : (kp == 32 ? 4 : 3);
  s.total = s.stages * kTileBytes + s.u_stages * kParts * s.u_bytes + s.g_stages * kParts * s.g_bytes + 512 + 1024;
  return s;
}

// A ring position and the parity of the round it is in
struct Ring {
  int i = 0;
  uint32_t round = 0;
  __device__ __forceinline__ void next(int n) {
    if (++i == n) {
      i = 0;
      round ^= 1u;
    }
  }
};

// What a quarter (32 rows) of row block `block` of a tensor is.  (rows and columns fit 32 bits)
struct Quarter {
  int map;          // tensor map of its weights
  int y;            // first row within the map
  int shift;        // column of the first whole octet
  int row;          // row of lane 0
  int whole;        // elements in whole octets of a row
  __device__ __forceinline__ Quarter(int cols, int block, int q) {
    if ((cols & 7) == 0) {
      map = 0;
      row = 128 * block + 32 * q;
      y = row;
      shift = 0;
      whole = cols;
    } else {
      map = 4 * (block & 1) + q;
      y = (block >> 1) * 32;
      row = (block >> 1) * 256 + map;
      shift = (-map * (cols & 7)) & 7;
      whole = (cols - shift) & ~7;
    }
  }
};
__device__ __forceinline__ int u_map(const TensorDesc& td) { return (td.cols & 7) ? 8 : 1; }
__device__ __forceinline__ int row_blocks(const WorkItem& w) { return static_cast<int>((w.nrows_or_count + 127) >> 7); }

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&v)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "r"(taddr)
               : "memory");
}

// Octet of the staged tile: 16 or 32 bytes of a 128-byte row whose chunks are swizzled (`row` = address of the row, xor16 = its
// swizzle).
template <typename T>
struct StagedOctet {
  static __device__ __forceinline__ void load(uint32_t row, uint32_t xor16, int o, float (&f)[8]) {
    const uint4 v = lds128(row + ((static_cast<uint32_t>(o) << 4) ^ xor16));
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if constexpr (std::is_same<T, __nv_bfloat16>::value) {
        f[2 * i] = __uint_as_float(w[i] << 16);
        f[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
      } else {
        const float2 h = __half22float2(*reinterpret_cast<const __half2*>(&w[i]));
        f[2 * i] = h.x;
        f[2 * i + 1] = h.y;
      }
    }
  }
  static __device__ __forceinline__ void store(uint32_t row, uint32_t xor16, int o, const float (&f)[8]) {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if constexpr (std::is_same<T, __nv_bfloat16>::value) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
        w[i] = *reinterpret_cast<const uint32_t*>(&h);
      } else {
        const __half2 h = __floats2half2_rn(f[2 * i], f[2 * i + 1]);
        w[i] = *reinterpret_cast<const uint32_t*>(&h);
      }
    }
    sts128(row + ((static_cast<uint32_t>(o) << 4) ^ xor16), make_uint4(w[0], w[1], w[2], w[3]));
  }
};
template <>
struct StagedOctet<float> {
  static __device__ __forceinline__ void load(uint32_t row, uint32_t xor16, int o, float (&f)[8]) {
    const uint4 a = lds128(row + ((static_cast<uint32_t>(o) << 5) ^ xor16)), b = lds128(row + (((static_cast<uint32_t>(o) << 5) + 16u) ^ xor16));
    f[0] = __uint_as_float(a.x); f[1] = __uint_as_float(a.y); f[2] = __uint_as_float(a.z); f[3] = __uint_as_float(a.w);
    f[4] = __uint_as_float(b.x); f[5] = __uint_as_float(b.y); f[6] = __uint_as_float(b.z); f[7] = __uint_as_float(b.w);
  }
  static __device__ __forceinline__ void store(uint32_t row, uint32_t xor16, int o, const float (&f)[8]) {
    sts128(row + ((static_cast<uint32_t>(o) << 5) ^ xor16),
           make_uint4(__float_as_uint(f[0]), __float_as_uint(f[1]), __float_as_uint(f[2]), __float_as_uint(f[3])));
    sts128(row + (((static_cast<uint32_t>(o) << 5) + 16u) ^ xor16),
           make_uint4(__float_as_uint(f[4]), __float_as_uint(f[5]), __float_as_uint(f[6]), __float_as_uint(f[7])));
  }
};

// One weight through L2: a line that this SM's L1 kept from before the previous kernel's stores would be stale.
template <typename T>
__device__ __forceinline__ float load_weight(const T* p) {
  if constexpr (sizeof(T) == 4) {
    return __ldcg(reinterpret_cast<const float*>(p));
  } else {
    const unsigned short raw = __ldcg(reinterpret_cast<const unsigned short*>(p));
    if constexpr (std::is_same<T, __nv_bfloat16>::value) return __uint_as_float(static_cast<uint32_t>(raw) << 16);
    else return __half2float(__ushort_as_half(raw));
  }
}

}  // namespace

template <typename T, int BITS, bool PRECISE, bool MULTI, bool SSTATS>
__global__ void __launch_bounds__(kThreadsStaged, 1) sweep_staged_kernel(const __grid_constant__ SweepParams p, int* __restrict__ error, const int kp) {
  using Cfg = StagedCfg<T>;
  constexpr int COLS = Cfg::COLS, HALF = Cfg::HALF, NSUB = Cfg::NSUB, NACC = Cfg::NACC, OCTS = HALF / 8;
  extern __shared__ uint8_t smem_raw[];
  const StagedSmem L = staged_smem(kp);
  const int S = L.stages, US = L.u_stages, GS = L.g_stages, rowb = L.rowb;
  uint8_t* theta_base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint8_t* u_base = theta_base + S * kTileBytes;
  uint8_t* g_base = u_base + US * kParts * L.u_bytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(g_base + GS * kParts * L.g_bytes);
  const uint32_t bar0 = smem_u32(bars);
  auto BAR_FULL = [&](int s) { return bar0 + 8u * static_cast<uint32_t>(s); };                                   // weights landed
  auto BAR_OUT = [&](int s) { return bar0 + 8u * static_cast<uint32_t>(kMaxStages + s); };                       // result written into the stage
  auto BAR_ACC_FULL = [&](int b) { return bar0 + 8u * static_cast<uint32_t>(2 * kMaxStages + b); };
  auto BAR_ACC_EMPTY = [&](int b) { return bar0 + 8u * static_cast<uint32_t>(2 * kMaxStages + 4 + b); };
  auto BAR_U_FULL = [&](int u) { return bar0 + 8u * static_cast<uint32_t>(2 * kMaxStages + 8 + u); };
  auto BAR_U_FREE = [&](int u) { return bar0 + 8u * static_cast<uint32_t>(2 * kMaxStages + 10 + u); };
  auto BAR_G = [&](int g) { return bar0 + 8u * static_cast<uint32_t>(2 * kMaxStages + 12 + g); };
  auto BAR_ITEM = [&](int i) { return bar0 + 8u * static_cast<uint32_t>(2 * kMaxStages + 14 + i); };             // item published
  auto BAR_ITEM_READ = [&](int i) { return bar0 + 8u * static_cast<uint32_t>(2 * kMaxStages + 14 + kRing + i); };   // read by the other roles
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kMaxStages + 14 + 2 * kRing);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* ring = abort_flag + 1;
  // Number of the CTA's n-th item, or n_items at the end (and when a wait gave up); called once per n by each reading thread or warp.
  auto item = [&](int n) -> int {
    if (!mbar_wait<false>(BAR_ITEM(n % kRing), (n / kRing) & 1, abort_flag, error, 36)) return p.n_items;
    return ring[n % kRing];
  };
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(BAR_FULL(s), 1);
      mbar_init(BAR_OUT(s), kGroupWarps);
    }
    for (int b = 0; b < NACC; ++b) {
      mbar_init(BAR_ACC_FULL(b), 1);
      mbar_init(BAR_ACC_EMPTY(b), kGroupWarps);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(BAR_U_FULL(i), 1);
      mbar_init(BAR_U_FREE(i), 1);
      mbar_init(BAR_G(i), kEpi);
    }
    for (int i = 0; i < kRing; ++i) {
      mbar_init(BAR_ITEM(i), 1);
      mbar_init(BAR_ITEM_READ(i), 1 + kEpi);
    }
    *abort_flag = 0;
    fence_mbar_init();
  }
  __syncthreads();
  if (warp == 1) {
    tmem_alloc(smem_u32(tmem_slot), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot + kTmemBase;
  if (warp == 1) dependency_begin(p);     // (warp 0: after the first item is out; the epilogue warps: after the first strip)

  // All roles walk the same sequence of (item, row block, tile).
  if (warp == 0) {
    // ------------------------------------------------ items, loads and stores
    // Lane l < 8 looks after box l of every tile: quarter l / 2, bytes 128 (l mod 2) ... of its rows (tensors of whole octets: lanes 0
    // and 1, boxes of 128 rows).  One thread for all of it took longer per tile than the epilogue does.
    const CUtensorMap* box_map[kMaxStages] = {};      // of the tile in each stage; null: nothing of this lane's there
    int box_x[kMaxStages] = {}, box_y[kMaxStages] = {};
    const uint32_t box_at = smem_u32(theta_base) + static_cast<uint32_t>((4 * (lane & 1) + (lane >> 1)) * kBoxBytes);
    auto store_box = [&](int s) {
      if (box_map[s] != nullptr) tma_store_2d(box_map[s], box_x[s], box_y[s], box_at + static_cast<uint32_t>(s * kTileBytes));
      tma_commit();
    };
    // Every lane waits itself: what it has seen completed is in order before the copies that it issues.  (Lane 0 waiting for all, with a
    // shuffle and __syncwarp(), is slower too: six RoBERTa-shaped fp32 layers of rank 32 786 / 771 us, 20 M bf16 weights of rank 8 108 / 104.)
    auto wait0 = [&](uint32_t bar, uint32_t parity, int where) -> bool { return __all_sync(0xFFFFFFFFu, mbar_wait<true>(bar, parity, abort_flag, error, where)); };
    Ring st, ur;
    int t = 0, rb = 0;
    bool ok = true;
    int it = p.starts ? p.starts[blockIdx.x] : static_cast<int>(blockIdx.x);
    const int share_end = p.starts ? p.starts[blockIdx.x + 1] : 0;
    for (int n = 0; ok; ++n) {
      if (n >= kRing && !wait0(BAR_ITEM_READ(n % kRing), ((n / kRing) - 1) & 1, 30)) break;
      if (lane == 0) {
        ring[n % kRing] = it;
        mbar_arrive(BAR_ITEM(n % kRing));
      }
      if (n == 0) dependency_begin(p);
      if (it >= p.n_items) break;
      const WorkItem w = p.items[it];
      // the next item (as in ItemFeed of the CUDA-core kernels: one fetch beyond the end per CTA, the last one resets)
      int after = p.n_items;
      if (p.starts) {
        if (it + 1 < share_end) after = it + 1;
      } else if (p.n_items > static_cast<int>(gridDim.x)) {
        int f = 0;
        if (lane == 0) {
          f = atomicAdd(p.sched, 1);
          if (f == p.n_items - 1) *p.sched = 0;
        }
        after = __shfl_sync(0xFFFFFFFFu, f, 0) + static_cast<int>(gridDim.x);
      }
      it = after;
      const TensorDesc& td = p.tensors[w.tensor];
      const int rows = static_cast<int>(td.rows), cols = static_cast<int>(td.cols);
      const bool parts = (cols & 7) != 0;
      const CUtensorMap* maps = static_cast<const CUtensorMap*>(td.maps);
      const CUtensorMap* umap = maps + u_map(td) + lane;
      const uint32_t box_bytes = parts ? kBoxBytes : 4 * kBoxBytes;
      const int block0 = static_cast<int>(w.row0_or_e0 >> 7), col0 = static_cast<int>(w.col0);
      const int blocks = row_blocks(w);
      for (int r = 0; r < blocks && ok; ++r, ++rb) {
        if (rb >= US && !wait0(BAR_U_FREE(ur.i), ur.round ^ 1u, 31)) { ok = false; break; }
        if (lane == 0) mbar_arrive_expect_tx(BAR_U_FULL(ur.i), static_cast<uint32_t>(kParts * L.u_bytes));
        __syncwarp();
        if (lane < kParts)
          tma_load_2d(smem_u32(u_base) + static_cast<uint32_t>((ur.i * kParts + lane) * L.u_bytes), umap, 0, (block0 + r) * 128, BAR_U_FULL(ur.i));
        ur.next(US);
        const Quarter qt(cols, block0 + r, (lane >> 1) & 3);
        const bool rows_here = lane < (parts ? 8 : 2) && qt.row < rows;
        for (int sub = 0; sub < NSUB && COLS * sub < w.ncols; ++sub, ++t) {
          const int s = st.i;
          if (t >= S) {
            // the epilogue has written tile t-S into this stage: store it, then the stage is free
            if (!wait0(BAR_OUT(s), st.round ^ 1u, 32)) { ok = false; break; }
            store_box(s);
            tma_wait_read0();
          }
          const int x = col0 + COLS * sub + HALF * (lane & 1);
          const bool mine = rows_here && x < qt.whole;
          box_map[s] = mine ? maps + qt.map : nullptr;
          box_x[s] = x;
          box_y[s] = qt.y;
          const uint32_t bytes = static_cast<uint32_t>(__popc(__ballot_sync(0xFFFFFFFFu, mine))) * box_bytes;
          if (lane == 0) mbar_arrive_expect_tx(BAR_FULL(s), bytes);
          __syncwarp();
          if (mine) tma_load_2d(box_at + static_cast<uint32_t>(s * kTileBytes), maps + qt.map, x, qt.y, BAR_FULL(s));
          st.next(S);
        }
      }
    }
    // drain: store the last tiles, oldest first
    for (int v = (t > S ? t - S : 0); v < t && ok; ++v) {
      if (!wait0(BAR_OUT(v % S), (v / S) & 1, 33)) { ok = false; break; }
      store_box(v % S);
    }
    __syncwarp();
    if (lane == 0) {
      // let the loads still in flight land before the CTA gives up its shared memory (weights: only when aborting)
      for (int v = (t > S ? t - S : 0); v < t && !ok; ++v) {
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
    __syncwarp();
    tma_wait_all0();
  } else if (warp == 1) {
    // ------------------------------------------------ products
    if (elect_one()) {
      const uint32_t idesc_whole = make_idesc(1, COLS), idesc_parts = make_idesc(1, COLS + 16);
      const uint64_t desc_u0 = make_desc(smem_u32(u_base), rowb);
      const uint64_t desc_g0 = make_desc(smem_u32(g_base), rowb);
      const uint64_t u_part = static_cast<uint64_t>(L.u_bytes >> 4), g_part = static_cast<uint64_t>(L.g_bytes >> 4);
      Ring ur, ar;
      int t = 0;
      bool ok = true;
      for (int item_no = 0; ok; ++item_no) {
        const int it = item(item_no);
        mbar_arrive(BAR_ITEM_READ(item_no % kRing));
        if (it >= p.n_items) break;
        const WorkItem w = p.items[it];
        const TensorDesc& td = p.tensors[w.tensor];
        const uint32_t idesc = (td.cols & 7) ? idesc_parts : idesc_whole;
        const int g = item_no % GS;
        if (!mbar_wait<true>(BAR_G(g), (item_no / GS) & 1, abort_flag, error, 34)) break;
        const int blocks = row_blocks(w);
        for (int r = 0; r < blocks && ok; ++r) {
          const int u = ur.i;
          if (!mbar_wait<true>(BAR_U_FULL(u), ur.round, abort_flag, error, 35)) { ok = false; break; }
          const uint64_t du = desc_u0 + static_cast<uint64_t>((u * kParts * L.u_bytes) >> 4);
          for (int sub = 0; sub < NSUB && COLS * sub < w.ncols; ++sub, ++t) {
            if (t >= NACC && !mbar_wait<true>(BAR_ACC_EMPTY(ar.i), ar.round ^ 1u, abort_flag, error, 37)) { ok = false; break; }
            tc_fence_after();
            const uint64_t dg = desc_g0 + static_cast<uint64_t>((g * kParts * L.g_bytes + sub * COLS * rowb) >> 4);
            const uint32_t d = tmem_base + static_cast<uint32_t>(ar.i * Cfg::ACC_COLS);
            // smallest products first: (0,2) (2,0) (1,1) (0,1) (1,0) (0,0); part 0 is the leading one
            uint32_t acc = 0;
#pragma unroll
            for (int pr = 0; pr < 6; ++pr) {
              constexpr int kA[6] = {0, 2, 1, 0, 1, 0}, kB[6] = {2, 0, 1, 1, 0, 0};
              for (int k = 0; k < kp / 16; ++k) {
                umma(d, du + kA[pr] * u_part + static_cast<uint64_t>(2 * k), dg + kB[pr] * g_part + static_cast<uint64_t>(2 * k), idesc, acc);
                acc = 1;
              }
            }
            umma_commit(BAR_ACC_FULL(ar.i));
            ar.next(NACC);
          }
          if (ok) umma_commit(BAR_U_FREE(u));   // arrives once every product that reads this U tile has completed
          ur.next(US);
        }
      }
    }
  } else {
    // ------------------------------------------------ epilogue
    const int e = warp - 2, et = e * 32 + lane;
    const int quad = warp & 3;                               // tensor-memory lanes 32 quad ..., the quarter of the tile
    const int grp = e / kGroupWarps, box = (e >> 2) & 1;     // which tiles: t % 2 == grp; which 128 bytes of their rows
    const uint32_t tmem_warp = tmem_base + (static_cast<uint32_t>(32 * quad) << 16) + static_cast<uint32_t>(HALF * box);
    const uint32_t theta_row = smem_u32(theta_base) + static_cast<uint32_t>((4 * box + quad) * kBoxBytes + lane * 128);
    const uint32_t xor16 = static_cast<uint32_t>(lane & 7) << 4;
    const uint32_t g_s = smem_u32(g_base);
    const uint32_t zero = static_cast<uint32_t>(p.early) >> 1;       // (early is 0 or 1; see normals8_acc_linked)
    Ring st, ar;
    int t = 0, item_no = 0;
    int seen = -1, before = -1;       // last tile whose products this warp has waited for; last tile of the item before this one
    bool ok = true;
    auto strip_for = [&](int it, int no) {
      const WorkItem w = p.items[it];
      const TensorDesc& td = p.tensors[w.tensor];
      build_strip<BITS, PRECISE, MULTI>(td, p, w.col0, (td.cols & 7) ? kTileN : 128, kp, rowb, L.g_bytes,
                                        g_s + static_cast<uint32_t>((no % GS) * kParts * L.g_bytes), et);
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(BAR_G(no % GS));
    };
    // The products up to tile v are complete (so that the strip they read may be overwritten).  Only asked for when no tile that
    // reuses the accumulator of v can have been begun: its strip is the one that is about to be made.
    auto products_done = [&](int v) -> bool {
      if (v <= seen) return true;
      return mbar_wait<false>(BAR_ACC_FULL(v % NACC), (v / NACC) & 1, abort_flag, error, 38);
    };
    auto take = [&](int n) -> int {
      const int it = item(n);
      __syncwarp();
      if (lane == 0) mbar_arrive(BAR_ITEM_READ(n % kRing));
      return it;
    };
    int it = take(0);
    // the first strip is made of the seed alone, unless codes are delivered for it, which may come from earlier work in the stream
    const bool codes = it < p.n_items && p.tensors[p.items[it].tensor].q != nullptr;
    if (codes) dependency_begin(p);
    if (it < p.n_items) strip_for(it, 0);
    if (!codes) dependency_begin(p);
    for (int it_next; it < p.n_items && ok; it = it_next, ++item_no) {
      it_next = p.n_items;
      const WorkItem w = p.items[it];
      const TensorDesc& td = p.tensors[w.tensor];
      const uint32_t tid = static_cast<uint32_t>(td.id);
      const int cols = static_cast<int>(td.cols), rows = static_cast<int>(td.rows);
      const bool parts = sizeof(T) == 2 && (cols & 7) != 0;  // rows that are no multiple of eight elements: 16-bit storage only
      const int stride = parts ? 8 : 1;                      // rows between neighbouring lanes
      T* const base = static_cast<T*>(td.data);
      const PhiloxPre pre = philox_pre(0u, tid, p.term[0].keys);     // (tensors of 2^34 elements and more are not served here)
      const int block0 = static_cast<int>(w.row0_or_e0 >> 7), col0 = static_cast<int>(w.col0), ncols = w.ncols;
      const int blocks = row_blocks(w);
      double s_iso = 0.0, s_gd = 0.0, s_z = 0.0;             // SSTATS only
      // The strip of the next item goes into the other buffer before this group's last tile of this item, so that its products run
      // while that one is worked on: in the last row block, or where that holds one tile, the other group's, in the one before it.
      // (16-bit matrices of a few row blocks, us a step against the last row block for both groups: 128 wide, rank 8, 8 M weights 59.2 / 57.2;
      // 512 wide, 13 M 60.4 / 57.5; 120 M ragged 465 / 456.  Several seeds on 100 M: 552 / 562, hence not there.)
      const int strip_at = NSUB == 2 || MULTI || GS == 1 || blocks == 1 || ((t + blocks - 1) & 1) == grp ? blocks - 1 : blocks - 2;
      for (int r = 0; r < blocks && ok; ++r) {
        if (r == strip_at) {
          it_next = take(item_no + 1);
          if (GS == 2 && it_next < p.n_items) {
            if (!products_done(before)) { ok = false; break; }
            strip_for(it_next, item_no + 1);
          }
        }
        for (int sub = 0; sub < NSUB && COLS * sub < ncols; ++sub, ++t, st.next(S), ar.next(NACC)) {
          if ((t & 1) != grp) continue;                      // the other group's tile
          const int s = st.i, b = ar.i;
          if (!mbar_wait<false>(BAR_ACC_FULL(b), ar.round, abort_flag, error, 39)) { ok = false; break; }
          seen = t;
          if (!mbar_wait<false>(BAR_FULL(s), st.round, abort_flag, error, 40)) { ok = false; break; }
          tc_fence_after();
          __syncwarp();
          const Quarter qt(cols, block0 + r, quad);
          if (qt.row < rows) {
            const int x0 = col0 + COLS * sub + HALF * box;                     // of the warp's first octet, from the first whole one of the row
            const int n_oct = min(OCTS, (qt.whole - x0) >> 3);                 // whole octets here (none: zero or less)
            const int row = qt.row + stride * lane;
            const int64_t row_e = static_cast<int64_t>(row) * cols;
            const uint32_t oct0 = static_cast<uint32_t>((row_e + qt.shift + x0) >> 3);
            const uint32_t tm = tmem_warp + static_cast<uint32_t>(b * Cfg::ACC_COLS + qt.shift);
            const uint32_t trow = theta_row + static_cast<uint32_t>(s * kTileBytes);
            // half the octets at a time: four (16-bit weights) or two (fp32), whose generator chains interleave
            constexpr int W = OCTS / 2;
#pragma unroll
            for (int o0 = 0; o0 < OCTS; o0 += W) {
              if (o0 >= n_oct) break;
              float z[W][8];
              {
                uint32_t h[W / 2][16];
#pragma unroll
                for (int i = 0; i < W / 2; ++i) tmem_ld16(tm + static_cast<uint32_t>(8 * o0 + 16 * i), h[i]);
                tmem_ld_wait();
#pragma unroll
                for (int x = 0; x < W; ++x)
#pragma unroll
                  for (int i = 0; i < 8; ++i) z[x][i] = __uint_as_float(h[x >> 1][8 * (x & 1) + i]);
              }
              const uint32_t oct = oct0 + static_cast<uint32_t>(o0);
              if constexpr (SSTATS) {
#pragma unroll
                for (int x = 0; x < W; ++x) {
                  float d[8], f_iso = 0.0f, f_gd = 0.0f, f_z = 0.0f;
#pragma unroll
                  for (int i = 0; i < 8; ++i) {
                    d[i] = z[x][i];
                    z[x][i] = 0.0f;
                  }
                  normals8_add<BITS, PRECISE>(p.term[0].keys, pre, oct + x, p.term[0].iso, z[x]);
#pragma unroll
                  for (int i = 0; i < 8; ++i) {
                    f_iso = fmaf(z[x][i], z[x][i], f_iso);
                    f_gd = fmaf(d[i], d[i], f_gd);
                    z[x][i] += d[i];
                    f_z = fmaf(z[x][i], z[x][i], f_z);
                  }
                  if (row < rows && o0 + x < n_oct) {
                    s_iso += static_cast<double>(f_iso);
                    s_gd += static_cast<double>(f_gd);
                    s_z += static_cast<double>(f_z);
                  }
                }
              } else {
                uint32_t link = 0;
#pragma unroll
                for (int x = 0; x < W; ++x) {
                  if constexpr (!PRECISE && BITS == 16) normals8_acc_linked(p.term[0].keys, pre, oct + x, p.term[0].iso, zero, link, z[x]);
                  else normals8_add<BITS, PRECISE>(p.term[0].keys, pre, oct + x, p.term[0].iso, z[x]);
                }
              }
              if (MULTI) {
#pragma unroll 1
                for (int q = 1; q < p.n_terms; ++q) {
                  const PhiloxKeys& keys = p.term[q].keys;
                  const PhiloxPre pre_q = philox_pre(0u, tid, keys);
                  uint32_t link = 0;
#pragma unroll
                  for (int x = 0; x < W; ++x) {
                    if constexpr (!PRECISE && BITS == 16) normals8_acc_linked(keys, pre_q, oct + x, p.term[q].iso, zero, link, z[x]);
                    else normals8_add<BITS, PRECISE>(keys, pre_q, oct + x, p.term[q].iso, z[x]);
                  }
                }
              }
#pragma unroll
              for (int x = 0; x < W; ++x) {
                float th[8];
                StagedOctet<T>::load(trow, xor16, o0 + x, th);
#pragma unroll
                for (int i = 0; i < 8; i += 2) unpack2(add2(pack2(th[i], th[i + 1]), pack2(z[x][i], z[x][i + 1])), th[i], th[i + 1]);
                StagedOctet<T>::store(trow, xor16, o0 + x, th);
              }
            }
            if (parts) {
              // the ends of the rows, element by element, 0: columns before the first whole octet, 1: behind the last one
              const bool head = qt.shift > 0 && x0 == 0, tail = qt.shift + qt.whole < cols && qt.whole >= x0 && qt.whole < x0 + HALF;
#pragma unroll 1
              for (int end = head ? 0 : 1; end < (tail ? 2 : 1); ++end) {
                const int c0 = end == 0 ? qt.shift - 8 : qt.shift + qt.whole;      // column of the octet's first element
                const int i0 = end == 0 ? 8 - qt.shift : 0, i1 = end == 0 ? 8 : cols - c0;
                uint32_t d[8];
                __syncwarp();
                tmem_ld8(tm + static_cast<uint32_t>(c0 - qt.shift - x0), d);
                tmem_ld_wait();
                if (row < rows) {
                  T* const at = base + (row_e + c0);
                  float th[8], z[8];
#pragma unroll
                  for (int i = 0; i < 8; ++i) th[i] = i >= i0 && i < i1 ? load_weight(at + i) : 0.0f;
                  // (the sums in the order of whole octets: the normals go onto the product, or both apart for their norms)
                  if constexpr (SSTATS) {
                    iso8<BITS, PRECISE, MULTI>(p, tid, static_cast<uint64_t>(row_e + c0), z);
                  } else {
                    const uint32_t oct = static_cast<uint32_t>((row_e + c0) >> 3);
#pragma unroll
                    for (int i = 0; i < 8; ++i) z[i] = __uint_as_float(d[i]);
                    normals8_add<BITS, PRECISE>(p.term[0].keys, pre, oct, p.term[0].iso, z);
                    if (MULTI) {
#pragma unroll 1
                      for (int q = 1; q < p.n_terms; ++q)
                        normals8_add<BITS, PRECISE>(p.term[q].keys, philox_pre(0u, tid, p.term[q].keys), oct, p.term[q].iso, z);
                    }
                  }
                  float f_iso = 0.0f, f_gd = 0.0f, f_z = 0.0f;
#pragma unroll
                  for (int i = 0; i < 8; ++i)
                    if (i >= i0 && i < i1) {
                      if constexpr (SSTATS) {
                        const float g = __uint_as_float(d[i]);
                        f_iso = fmaf(z[i], z[i], f_iso);
                        f_gd = fmaf(g, g, f_gd);
                        z[i] += g;
                        f_z = fmaf(z[i], z[i], f_z);
                      }
                      Storage<T>::store1(at + i, th[i] + z[i]);
                    }
                  s_iso += static_cast<double>(f_iso);
                  s_gd += static_cast<double>(f_gd);
                  s_z += static_cast<double>(f_z);
                }
                __syncwarp();
              }
            }
          }
          tc_fence_before();
          fence_proxy_async();
          __syncwarp();
          if (lane == 0) {
            mbar_arrive(BAR_ACC_EMPTY(b));
            mbar_arrive(BAR_OUT(s));
          }
        }
      }
      if (GS == 1 && it_next < p.n_items && ok) {
        if (!products_done(t - 1)) { ok = false; break; }
        strip_for(it_next, item_no + 1);
      }
      before = t - 1;
      if constexpr (SSTATS) {
        if (ok) store_item_stats(p, it, e, s_iso, s_gd, s_z);
      }
    }
  }

  // ---- common exit ----
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base - kTmemBase, 512);
  }
}

namespace {
template <typename T, int BITS, bool PRECISE, bool MULTI, bool SSTATS>
cudaError_t launch_staged_one(int kp, const SweepParams& p, int* error, int grid, cudaStream_t st) {
  auto k = sweep_staged_kernel<T, BITS, PRECISE, MULTI, SSTATS>;
  const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448);
  if (e != cudaSuccess) return e;
  return launch_sweep_kernel(k, grid, kThreadsStaged, static_cast<size_t>(staged_smem(kp).total), st, p, error, kp);
}
template <typename T, bool PRECISE>
cudaError_t launch_staged_typed(const KernelChoice& kc, const SweepParams& p, int* error, int grid, cudaStream_t st) {
  if (p.n_terms > 1)
    return kc.bits == 32 ? launch_staged_one<T, 32, PRECISE, true, false>(kc.kpad, p, error, grid, st)
                         : launch_staged_one<T, 16, PRECISE, true, false>(kc.kpad, p, error, grid, st);
  if (p.item_stats != nullptr)
    return kc.bits == 32 ? launch_staged_one<T, 32, PRECISE, false, true>(kc.kpad, p, error, grid, st)
                         : launch_staged_one<T, 16, PRECISE, false, true>(kc.kpad, p, error, grid, st);
  return kc.bits == 32 ? launch_staged_one<T, 32, PRECISE, false, false>(kc.kpad, p, error, grid, st)
                       : launch_staged_one<T, 16, PRECISE, false, false>(kc.kpad, p, error, grid, st);
}
}  // namespace

cudaError_t launch_sweep_staged(const KernelChoice& kc, const SweepParams& p, int* error, int grid, cudaStream_t st) {
  static_assert(kEpi <= kStatSlots, "one bookkeeping slot per epilogue warp");
  switch (kc.dtype) {
    case 0: return launch_staged_typed<float, true>(kc, p, error, grid, st);
    case 1: return launch_staged_typed<__half, false>(kc, p, error, grid, st);
    case 2: return launch_staged_typed<__nv_bfloat16, false>(kc, p, error, grid, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace zgr
