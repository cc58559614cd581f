// Sweep with a tensor-core contraction for the guided tensors that neither TMA-staged kernel (zgr_umma.cu, zgr_staged.cu) takes: fp32
// rows that are no multiple of eight elements long, weights that do not begin on a 16-byte boundary, rows shorter than two
// octets, and small sets (tensor_core_kind and staged_kind in zgr_host.cu have the sizes).
//     theta <- rnd(theta + c (a Z + b U G))            (Eq. (perturbation) applied as in Algorithm 1)
//
// Layout.  Generator blocks run along the flattened tensor, eight elements ("an octet") at a time, so in a tensor whose
// row length is no multiple of eight the octets of row m start at column  h_m = -(m cols) mod 8  and one of them
// straddles each row end.  A work item is a strip of 128 columns x a range of rows; within it a row owns the
// octets whose first element falls into the strip (16 of them, whatever h_m is), plus, in the strip at column 0, the
// tail of the octet that began in the row before.  An owned octet reaches up to 7 columns beyond the strip, so the
// product tile is computed 144 columns wide.
//
// Pipeline (one CTA per SM; small sets give it a contiguous share of the items, otherwise its first item is its own index and
// the others come from a counter in global memory):
//   warp 0   hands out the items through a ring of four, TMA loads of U, 128 rows at a time, pre-split into three bf16 parts
//   warp 1   tcgen05.mma:  D = c b U G  (128 x 144, fp32) into one of three tensor-memory buffers
//   warps 2-17  coefficient strips c b G (three bf16 parts, K-major) into shared memory, one item ahead where two strips
//            fit; then per tile and warp 32 rows x 32 columns: D through a warp-private shared-memory buffer, from one
//            row per thread (tensor memory) to one octet per thread (global memory: four lanes take 64 / 128
//            contiguous bytes of a row), and there the weights are loaded, the normals added, the result rounded and stored.
//
// Operand precision.  An fp32 number is the sum of three bf16 numbers (8 bits each) without error and without range
// limits; six of the nine products are formed, the others are below 2^-24 of the result.  With the copies of U leaning against
// the truncation of the tensor cores (truncation_lean) the contraction is as accurate as a chain of fp32 multiply-adds, from
// rank 2 on more so.
//
// Bank conflicts of the transposition.  Row m of a warp's buffer is `pitch` floats long; lane (m, o) reads
// D[m][h_m + 8 o + i].  Eight rows x four octets per read: distinct banks if m pitch + h_m = m (pitch - cols) takes
// eight different values modulo 8, i.e. if pitch - cols is odd.  pitch = 41 for an even, 42 for an odd number of columns
// (the writes, one float per row, are then at most two-way).  With cols a multiple of 8 every h_m is 0 and both sides
// use 128-bit accesses with pitch 36.
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

constexpr int kTileM = 128;
constexpr int kAcc = 3;                        // accumulator buffers: 3 x 144 of the 512 tensor-memory columns
constexpr int kTileThreads = 32 * (2 + kEpi);
constexpr int kRing = 4;                       // items published ahead
constexpr int kPitchMax = 42;
constexpr int kXposeBytes = 32 * kPitchMax * 4;   // one warp's buffer

// Shared-memory plan for contraction width kp (16, 32, 64).
struct TileSmem {
  int rowb, u_bytes, g_bytes, u_stages, g_stages, total;
};
__host__ __device__ inline TileSmem tile_smem(int kp) {
  TileSmem t;
  t.rowb = 2 * kp;
  t.u_bytes = kTileM * t.rowb;
  t.g_bytes = kTileN * t.rowb;
  t.u_stages = kp == 64 ? 1 : 2;               // width 64: one U tile and one strip fit beside the buffers
  t.g_stages = kp == 64 ? 1 : 2;
  t.total = t.u_stages * kParts * t.u_bytes + t.g_stages * kParts * t.g_bytes + kEpi * kXposeBytes + 256 + 1024;
  return t;
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[40]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,"
      "%29,%30,%31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]),
        "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]),
        "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld8_tail(uint32_t taddr, uint32_t (&v)[40]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(v[32]), "=r"(v[33]), "=r"(v[34]), "=r"(v[35]), "=r"(v[36]), "=r"(v[37]), "=r"(v[38]), "=r"(v[39])
               : "r"(taddr)
               : "memory");
}

// storage of an octet as it is loaded: 16 bytes of 16-bit weights, unpacked on use, or eight floats
template <typename T>
struct RawOct {
  uint4 v;
  __device__ __forceinline__ void load(const T* p, bool) { v = __ldcs(reinterpret_cast<const uint4*>(p)); }
  __device__ __forceinline__ void unpack(float (&f)[8]) const {
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
};
template <>
struct RawOct<float> {
  float v[8];
  __device__ __forceinline__ void load(const float* p, bool wide) { Storage<float>::load8(p, v, wide); }
  __device__ __forceinline__ void unpack(float (&f)[8]) const {
#pragma unroll
    for (int i = 0; i < 8; ++i) f[i] = v[i];
  }
};

}  // namespace

template <typename T, int BITS, bool PRECISE, bool MULTI, bool SSTATS>
__global__ void __launch_bounds__(kTileThreads, 1) sweep_tile_kernel(const __grid_constant__ SweepParams p, const CUtensorMap* __restrict__ tmaps,
                                                                     int* __restrict__ error, const int kp, const int by_residue) {
  extern __shared__ uint8_t smem_raw[];
  const TileSmem L = tile_smem(kp);
  const int US = L.u_stages, GS = L.g_stages, rowb = L.rowb;
  uint8_t* u_base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint8_t* g_base = u_base + US * kParts * L.u_bytes;
  uint8_t* x_base = g_base + GS * kParts * L.g_bytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(x_base + kEpi * kXposeBytes);
  const uint32_t bar0 = smem_u32(bars);
  auto BAR_ACC_FULL = [&](int b) { return bar0 + 8u * static_cast<uint32_t>(b); };
  auto BAR_ACC_EMPTY = [&](int b) { return bar0 + 8u * static_cast<uint32_t>(kAcc + b); };
  auto BAR_U_FULL = [&](int u) { return bar0 + 8u * static_cast<uint32_t>(2 * kAcc + u); };
  auto BAR_U_FREE = [&](int u) { return bar0 + 8u * static_cast<uint32_t>(2 * kAcc + 2 + u); };
  auto BAR_G = [&](int g) { return bar0 + 8u * static_cast<uint32_t>(2 * kAcc + 4 + g); };
  auto BAR_ITEM = [&](int i) { return bar0 + 8u * static_cast<uint32_t>(2 * kAcc + 6 + i); };            // item published
  auto BAR_ITEM_READ = [&](int i) { return bar0 + 8u * static_cast<uint32_t>(2 * kAcc + 6 + kRing + i); };   // read by the other roles
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kAcc + 6 + 2 * kRing);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* ring = abort_flag + 1;
  // Number of the CTA's n-th item, or n_items at the end (and when a wait gave up); called once per n by each reading thread or warp.
  auto item = [&](int n) -> int {
    if (!mbar_wait<false>(BAR_ITEM(n % kRing), (n / kRing) & 1, abort_flag, error, 26)) return p.n_items;
    return ring[n % kRing];
  };
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int b = 0; b < kAcc; ++b) {
      mbar_init(BAR_ACC_FULL(b), 1);
      mbar_init(BAR_ACC_EMPTY(b), kEpi);
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
  const uint32_t tmem_base = *tmem_slot;
  if (warp == 1) dependency_begin(p);     // (warp 0: after the first item is out; the epilogue warps: after the first strip)

  // All roles walk the same sequence of (item, row tile) pairs; t counts tiles over the life of the CTA.
  if (warp == 0) {
    // ------------------------------------------------ U loads
    if (elect_one()) {
      int t = 0;
      bool ok = true;
      int it = p.starts ? p.starts[blockIdx.x] : static_cast<int>(blockIdx.x);
      const int share_end = p.starts ? p.starts[blockIdx.x + 1] : 0;
      for (int n = 0; ok; ++n) {
        if (n >= kRing && !mbar_wait<true>(BAR_ITEM_READ(n % kRing), ((n / kRing) - 1) & 1, abort_flag, error, 20)) break;
        ring[n % kRing] = it;
        mbar_arrive(BAR_ITEM(n % kRing));
        if (n == 0) dependency_begin(p);
        if (it >= p.n_items) break;
        // the next item (as in ItemFeed of the CUDA-core kernels: one fetch beyond the end per CTA, the last one resets)
        int after = p.n_items;
        if (p.starts) {
          if (it + 1 < share_end) after = it + 1;
        } else if (p.n_items > static_cast<int>(gridDim.x)) {
          const int f = atomicAdd(p.sched, 1);
          if (f == p.n_items - 1) *p.sched = 0;
          after = f + static_cast<int>(gridDim.x);
        }
        const WorkItem w = p.items[it];
        it = after;
        const CUtensorMap* tm = tmaps + 3 * w.tensor;
        const int row_end = static_cast<int>(w.row0_or_e0 + w.nrows_or_count);
        for (int row0 = static_cast<int>(w.row0_or_e0); row0 < row_end; row0 += kTileM, ++t) {
          const int u = t % US;
          if (t >= US && !mbar_wait<true>(BAR_U_FREE(u), ((t / US) - 1) & 1, abort_flag, error, 21)) { ok = false; break; }
          const uint32_t dst = smem_u32(u_base + u * kParts * L.u_bytes);
          mbar_arrive_expect_tx(BAR_U_FULL(u), static_cast<uint32_t>(kParts * L.u_bytes));
          // (rows kept by residue for the staged kernel: the map puts them back in order, eight residues x 16)
          for (int i = 0; i < kParts; ++i) {
            if (by_residue) tma_load_4d(dst + i * L.u_bytes, tm + i, 0, 0, (row0 & 255) >> 3, row0 >> 8, BAR_U_FULL(u));
            else tma_load_2d(dst + i * L.u_bytes, tm + i, 0, row0, BAR_U_FULL(u));
          }
        }
      }
      // let the last loads land before the CTA gives up its shared memory
      for (int v = (t > US ? t - US : 0); v < t; ++v) {
        const unsigned long long t0 = clock64();
        while (!mbar_try_wait(BAR_U_FULL(v % US), (v / US) & 1) && clock64() - t0 < kWaitLimitCycles) {
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------ products
    if (elect_one()) {
      const uint32_t idesc = make_idesc(1, kTileN);
      const uint64_t desc_u0 = make_desc(smem_u32(u_base), rowb);
      const uint64_t desc_g0 = make_desc(smem_u32(g_base), rowb);
      const uint64_t u_part = static_cast<uint64_t>(L.u_bytes >> 4), g_part = static_cast<uint64_t>(L.g_bytes >> 4);
      int t = 0;
      bool ok = true;
      for (int item_no = 0; ok; ++item_no) {
        const int it = item(item_no);
        mbar_arrive(BAR_ITEM_READ(item_no % kRing));
        if (it >= p.n_items) break;
        const WorkItem w = p.items[it];
        const int g = item_no % GS;
        if (!mbar_wait<true>(BAR_G(g), (item_no / GS) & 1, abort_flag, error, 22)) break;
        const uint64_t dg = desc_g0 + static_cast<uint64_t>((g * kParts * L.g_bytes) >> 4);
        const int row_end = static_cast<int>(w.row0_or_e0 + w.nrows_or_count);
        for (int row0 = static_cast<int>(w.row0_or_e0); row0 < row_end; row0 += kTileM, ++t) {
          const int u = t % US, b = t % kAcc;
          if (!mbar_wait<true>(BAR_U_FULL(u), (t / US) & 1, abort_flag, error, 23)) { ok = false; break; }
          if (t >= kAcc && !mbar_wait<true>(BAR_ACC_EMPTY(b), ((t / kAcc) - 1) & 1, abort_flag, error, 24)) { ok = false; break; }
          tc_fence_after();
          const uint64_t du = desc_u0 + static_cast<uint64_t>((u * kParts * L.u_bytes) >> 4);
          const uint32_t d = tmem_base + static_cast<uint32_t>(b * kTileN);
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
          umma_commit(BAR_ACC_FULL(b));
          umma_commit(BAR_U_FREE(u));
        }
      }
    }
  } else {
    // ------------------------------------------------ epilogue
    const int e = warp - 2, et = e * 32 + lane;
    const int quad = warp & 3, cg = e >> 2;                  // tensor-memory lanes 32 quad ..., columns 32 cg ... of the strip
    const int sub = lane >> 2, o = lane & 3;                 // octet view: row 8 pass + sub, octet o of the 32 columns
    const uint32_t xbuf = smem_u32(x_base) + static_cast<uint32_t>(e * kXposeBytes);
    const uint32_t g_s = smem_u32(g_base);
    const uint32_t tmem_warp = tmem_base + (static_cast<uint32_t>(32 * quad) << 16) + static_cast<uint32_t>(32 * cg);
    int t = 0, item_no = 0;
    bool ok = true;
    auto strip_for = [&](int it, int no) {
      const WorkItem w = p.items[it];
      build_strip<BITS, PRECISE, MULTI>(p.tensors[w.tensor], p, w.col0, kTileN, kp, rowb, L.g_bytes, g_s + static_cast<uint32_t>((no % GS) * kParts * L.g_bytes), et);
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(BAR_G(no % GS));
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
      const int64_t cols = td.cols;
      const uint32_t cols8 = static_cast<uint32_t>(cols) & 7u;
      const bool even8 = cols8 == 0;
      const int pitch = even8 ? 36 : ((cols & 1) ? 42 : 41);
      T* const base = static_cast<T*>(td.data);
      const bool vec = (reinterpret_cast<uintptr_t>(base) & 15) == 0, wide = (reinterpret_cast<uintptr_t>(base) & 31) == 0;
      const int64_t row_end = w.row0_or_e0 + w.nrows_or_count;
      const int c_chunk = 32 * cg;                           // first column of this warp's chunk within the strip
      double s_iso = 0.0, s_gd = 0.0, s_z = 0.0;             // SSTATS only
      for (int64_t row0 = w.row0_or_e0; row0 < row_end && ok; row0 += kTileM, ++t) {
        // the strip of the next item goes into the other buffer before this item's last tile, so that its products run
        // while this tile is worked on
        if (row0 + kTileM >= row_end) {
          it_next = take(item_no + 1);
          if (GS == 2 && it_next < p.n_items) strip_for(it_next, item_no + 1);
        }
        const int b = t % kAcc;
        const int64_t wrow = row0 + 32 * quad;               // first row of this warp
        // one octet per pass: element index of its start, its column, the elements of it that belong to this row
        const uint32_t h_sub = (0u - static_cast<uint32_t>((wrow + sub) & 7) * cols8) & 7u;   // the same for all passes: rows 8 apart
        const int64_t e_sub = (wrow + sub) * cols + w.col0 + c_chunk + 8 * o + h_sub;
        const int64_t c = w.col0 + c_chunk + 8 * o + h_sub;
        const int n_el = static_cast<int>(min(static_cast<int64_t>(8), cols - c));
        const bool full = vec && n_el == 8;
        // weights of the first passes, on their way while the accumulator is waited for (four octets of 16-bit weights fit
        // the register budget, two of fp32)
        constexpr int kAhead = sizeof(T) == 4 ? 2 : 4;
        constexpr bool kPrefetchNext = sizeof(T) == 4;
        RawOct<T> raw[kAhead];
        auto fetch = [&](int pass, RawOct<T>& into) {
          if (full && wrow + 8 * pass + sub < row_end) into.load(base + e_sub + 8 * pass * cols, wide);
        };
#pragma unroll
        for (int pass = 0; pass < kAhead; ++pass) fetch(pass, raw[pass]);
        if constexpr (kPrefetchNext) {
          // the same octets of the next row tile: on their way from HBM to L2 while this one is worked on
          if (n_el > 0) {
#pragma unroll
            for (int pass = 0; pass < 4; ++pass)
              if (wrow + kTileM + 8 * pass + sub < row_end)
                asm volatile("prefetch.global.L2 [%0];" ::"l"(base + e_sub + (kTileM + 8 * pass) * cols));
          }
        }
        if (!mbar_wait<false>(BAR_ACC_FULL(b), (t / kAcc) & 1, abort_flag, error, 25)) { ok = false; break; }
        tc_fence_after();
        {
          uint32_t v[40];
          tmem_ld32(tmem_warp + static_cast<uint32_t>(b * kTileN), v);
          tmem_ld8_tail(tmem_warp + static_cast<uint32_t>(b * kTileN + 32), v);
          tmem_ld_wait();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(BAR_ACC_EMPTY(b));
          const uint32_t xrow = xbuf + static_cast<uint32_t>(lane * pitch * 4);
          if (even8) {
#pragma unroll
            for (int i = 0; i < 8; ++i) sts128(xrow + 16u * i, make_uint4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]));
          } else {
#pragma unroll
            for (int i = 0; i < 40; ++i) sts32(xrow + 4u * i, v[i]);
          }
        }
        __syncwarp();
        auto finish = [&](int64_t el, int i0, int i1, const float (&d)[8]) {
          const bool whole = vec && i0 == 0 && i1 == 8;
          float th[8], z[8];
          if (whole) {
            Storage<T>::load8(base + el, th);
          } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) th[i] = (i >= i0 && i < i1) ? Storage<T>::load1(base + el + i) : 0.0f;
          }
          if constexpr (!PRECISE && !SSTATS) {
            const uint64_t oct = static_cast<uint64_t>(el) >> 3;
#pragma unroll
            for (int i = 0; i < 8; ++i) z[i] = d[i];
            normals8_acc<BITS>(p.term[0].keys, tid, static_cast<uint32_t>(oct), static_cast<uint32_t>(oct >> 32), p.term[0].iso, z);
            if (MULTI) {
#pragma unroll 1
              for (int q = 1; q < p.n_terms; ++q)
                normals8_acc<BITS>(p.term[q].keys, tid, static_cast<uint32_t>(oct), static_cast<uint32_t>(oct >> 32), p.term[q].iso, z);
            }
          } else {
            iso8<BITS, PRECISE, MULTI>(p, tid, static_cast<uint64_t>(el), z);
            if (SSTATS) {
              float f_iso = 0.0f, f_gd = 0.0f, f_z = 0.0f;
#pragma unroll
              for (int i = 0; i < 8; ++i) {
                if (whole || (i >= i0 && i < i1)) {
                  f_iso = fmaf(z[i], z[i], f_iso);
                  f_gd = fmaf(d[i], d[i], f_gd);
                  f_z = fmaf(z[i] + d[i], z[i] + d[i], f_z);
                }
              }
              s_iso += static_cast<double>(f_iso);
              s_gd += static_cast<double>(f_gd);
              s_z += static_cast<double>(f_z);
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) z[i] += d[i];
          }
#pragma unroll
          for (int i = 0; i < 8; ++i) th[i] += z[i];
          if (whole) {
            Storage<T>::store8(base + el, th);
          } else {
#pragma unroll
            for (int i = 0; i < 8; ++i)
              if (i >= i0 && i < i1) Storage<T>::store1(base + el + i, th[i]);
          }
        };
        auto read_d = [&](int pass, float (&d)[8]) {
          const uint32_t xat = xbuf + static_cast<uint32_t>(((8 * pass + sub) * pitch + 8 * o + static_cast<int>(h_sub)) * 4);
          if (even8) {
            const uint4 d0 = lds128(xat), d1 = lds128(xat + 16);
            d[0] = __uint_as_float(d0.x); d[1] = __uint_as_float(d0.y); d[2] = __uint_as_float(d0.z); d[3] = __uint_as_float(d0.w);
            d[4] = __uint_as_float(d1.x); d[5] = __uint_as_float(d1.y); d[6] = __uint_as_float(d1.z); d[7] = __uint_as_float(d1.w);
          } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) d[i] = lds32(xat + 4u * i);
          }
        };
        // All octets of the warp whole and under one high counter word (nearly always): straight-line code, several octets
        // per thread whose generator chains interleave.  Otherwise (row ends, last rows) one octet after the other.
        constexpr int kShift = BITS == 32 ? 34 : 35;       // element index -> high word of its block number
        const uint32_t hi0 = static_cast<uint32_t>(static_cast<uint64_t>(e_sub) >> kShift);
        const bool fast = __all_sync(0xFFFFFFFFu, full && wrow + 24 + sub < row_end &&
                                                                 hi0 == static_cast<uint32_t>(static_cast<uint64_t>(e_sub + 24 * cols) >> kShift));
        if (fast) {
          const PhiloxPre pre = philox_pre(hi0, tid, p.term[0].keys);
          // as many at a time as were loaded ahead (a loop that is not unrolled: the accurate transform would fill the
          // instruction cache)
          constexpr int kWide = kAhead;
#pragma unroll 1
          for (int p0 = 0; p0 < 4; p0 += kWide) {
            float z[kWide][8];
            uint32_t oct[kWide];
#pragma unroll
            for (int x = 0; x < kWide; ++x) {
              read_d(p0 + x, z[x]);
              oct[x] = static_cast<uint32_t>(static_cast<uint64_t>(e_sub + 8 * (p0 + x) * cols) >> 3);
            }
            if constexpr (SSTATS) {
#pragma unroll
              for (int x = 0; x < kWide; ++x) {
                float d[8], f_iso = 0.0f, f_gd = 0.0f, f_z = 0.0f;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                  d[i] = z[x][i];
                  z[x][i] = 0.0f;
                }
                normals8_add<BITS, PRECISE>(p.term[0].keys, pre, oct[x], p.term[0].iso, z[x]);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                  f_iso = fmaf(z[x][i], z[x][i], f_iso);
                  f_gd = fmaf(d[i], d[i], f_gd);
                  z[x][i] += d[i];
                  f_z = fmaf(z[x][i], z[x][i], f_z);
                }
                s_iso += static_cast<double>(f_iso);
                s_gd += static_cast<double>(f_gd);
                s_z += static_cast<double>(f_z);
              }
            } else {
#pragma unroll
              for (int x = 0; x < kWide; ++x) normals8_add<BITS, PRECISE>(p.term[0].keys, pre, oct[x], p.term[0].iso, z[x]);
            }
            if (MULTI) {
#pragma unroll 1
              for (int q = 1; q < p.n_terms; ++q) {
                const PhiloxPre pre_q = philox_pre(hi0, tid, p.term[q].keys);
#pragma unroll
                for (int x = 0; x < kWide; ++x) normals8_add<BITS, PRECISE>(p.term[q].keys, pre_q, oct[x], p.term[q].iso, z[x]);
              }
            }
#pragma unroll
            for (int x = 0; x < kWide; ++x) {
              float th[8];
              raw[x].unpack(th);
#pragma unroll
              for (int i = 0; i < 8; ++i) th[i] += z[x][i];
              Storage<T>::store8(base + e_sub + 8 * (p0 + x) * cols, th, wide);
              if (p0 + kWide < 4) fetch(p0 + x + kWide, raw[x]);
            }
          }
        }
        // pass 4: the columns before the first octet of each row (lane = row), the tail of an octet that began in the previous row
        const bool head = !even8 && w.col0 == 0 && cg == 0;
#pragma unroll 1
        for (int pass = fast ? 4 : 0; pass < (head ? 5 : 4); ++pass) {
          float d[8];
          int64_t el = e_sub + 8 * pass * cols;
          int i0 = 0, i1 = wrow + 8 * pass + sub < row_end ? n_el : 0;
          if (pass < 4) {
            read_d(pass, d);
          } else {
            const int64_t row = wrow + lane;
            const int h = static_cast<int>((0u - static_cast<uint32_t>(row & 7) * cols8) & 7u);
            el = row * cols + h - 8;
            i0 = 8 - h;
            i1 = row < row_end && h > 0 ? static_cast<int>(min(static_cast<int64_t>(8), 8 - h + cols)) : 0;
#pragma unroll
            for (int i = 0; i < 8; ++i) d[i] = i >= i0 ? lds32(xbuf + static_cast<uint32_t>((lane * pitch + i - i0) * 4)) : 0.0f;
          }
          if (i1 > i0) finish(el, i0, i1, d);
        }
        __syncwarp();
      }
      if (GS == 1 && it_next < p.n_items && ok) strip_for(it_next, item_no + 1);   // every product that read the old strip has completed
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
    tmem_dealloc(tmem_base, 512);
  }
}

namespace {
template <typename T, int BITS, bool PRECISE, bool MULTI, bool SSTATS>
cudaError_t launch_tile_one(int kp, int by_residue, const SweepParams& p, const CUtensorMap* tmaps, int* error, int grid, cudaStream_t st) {
  auto k = sweep_tile_kernel<T, BITS, PRECISE, MULTI, SSTATS>;
  const int smem = tile_smem(kp).total;
  const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, tile_smem(64).total);
  if (e != cudaSuccess) return e;
  return launch_sweep_kernel(k, grid, kTileThreads, static_cast<size_t>(smem), st, p, tmaps, error, kp, by_residue);
}
template <typename T, bool PRECISE>
cudaError_t launch_tile_typed(const KernelChoice& kc, const SweepParams& p, const CUtensorMap* tmaps, int* error, int grid, cudaStream_t st) {
  if (p.n_terms > 1)
    return kc.bits == 32 ? launch_tile_one<T, 32, PRECISE, true, false>(kc.kpad, kc.by_residue, p, tmaps, error, grid, st)
                         : launch_tile_one<T, 16, PRECISE, true, false>(kc.kpad, kc.by_residue, p, tmaps, error, grid, st);
  if (p.item_stats != nullptr)
    return kc.bits == 32 ? launch_tile_one<T, 32, PRECISE, false, true>(kc.kpad, kc.by_residue, p, tmaps, error, grid, st)
                         : launch_tile_one<T, 16, PRECISE, false, true>(kc.kpad, kc.by_residue, p, tmaps, error, grid, st);
  return kc.bits == 32 ? launch_tile_one<T, 32, PRECISE, false, false>(kc.kpad, kc.by_residue, p, tmaps, error, grid, st)
                       : launch_tile_one<T, 16, PRECISE, false, false>(kc.kpad, kc.by_residue, p, tmaps, error, grid, st);
}
}  // namespace

cudaError_t launch_sweep_tile(const KernelChoice& kc, const SweepParams& p, const CUtensorMap* tmaps, int* error, int grid, cudaStream_t st) {
  static_assert(kEpi <= kStatSlots, "one bookkeeping slot per epilogue warp");
  switch (kc.dtype) {
    case 0: return launch_tile_typed<float, true>(kc, p, tmaps, error, grid, st);
    case 1: return launch_tile_typed<__half, false>(kc, p, tmaps, error, grid, st);
    case 2: return launch_tile_typed<__nv_bfloat16, false>(kc, p, tmaps, error, grid, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace zgr
