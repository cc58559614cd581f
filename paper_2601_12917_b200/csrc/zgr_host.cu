// Host side of the ZGR library: context, validation, work planning and the C entry points
// declared in include/zgr.h.  Everything numerical happens in the kernels; the host only
// combines the step scalars in double (Eq. (grad), Eq. (perturbation)) and hands them over as fp32.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <numeric>
#include <vector>

#include "zgr.h"
#include "zgr_internal.h"
#include "zgr_host_internal.h"
#include "zgr_kernels.h"
#include "zgr_subspace.h"

using namespace zgr;

namespace {

struct Group {
  KernelChoice kc;
  std::vector<WorkItem> items;
  WorkItem* d_items = nullptr;
  std::vector<int32_t> starts;                            // small tensor-core groups: first item of every CTA's share, and the end (else empty)
  int32_t* d_starts = nullptr;
  int grid = 0;
  int64_t elements = 0;                                   // weights covered by one launch
  double* d_item_stats = nullptr;                         // kStatSlots x 3 doubles per item (norm bookkeeping), allocated on first use
  int32_t* d_sched = nullptr;                             // CUDA-core and three-part kernels: two item counters (caller's stream, library's second stream)
  std::vector<int32_t> first_item;                        // per tensor l: index of its first item in `items` (size n + 1; items are in tensor order)
  std::vector<std::pair<cudaEvent_t, cudaEvent_t>> timed;  // per-launch events while profiling is on
};

int dtype_bytes(int dt) { return dt == ZGR_F32 ? 4 : 2; }

// Host-mapped status words of zgr_build_subspace, one per context that has called it, from one 16 KB page per process: pinning
// memory takes 1.2 to 2.8 ms, ten times a first call without it.  A word goes back when its context ends (no kernel writes it
// any more: the call waits for its kernel).  Beyond the page's 256 words a context pins its own.
class StatusWords {
  static constexpr int kWords = 256, kStride = 64 / sizeof(int);
  std::mutex mutex_;
  int* page_ = nullptr;
  bool used_[kWords] = {};

 public:
  cudaError_t take(int** word, bool* own) {
    const std::lock_guard<std::mutex> lock(mutex_);
    *own = false;
    if (page_ == nullptr) {
      void* page = nullptr;
      const cudaError_t e = cudaHostAlloc(&page, kWords * kStride * sizeof(int), cudaHostAllocMapped | cudaHostAllocPortable);
      if (e != cudaSuccess) return e;
      page_ = static_cast<int*>(page);
    }
    for (int i = 0; i < kWords; ++i)
      if (!used_[i]) {
        used_[i] = true;
        *word = page_ + i * kStride;
        return cudaSuccess;
      }
    *own = true;
    return cudaHostAlloc(reinterpret_cast<void**>(word), sizeof(int), cudaHostAllocMapped);
  }
  void give_back(int* word, bool own) {
    if (word == nullptr) return;
    if (own) {
      cudaFreeHost(word);
      return;
    }
    const std::lock_guard<std::mutex> lock(mutex_);
    used_[(word - page_) / kStride] = false;
  }
};
StatusWords& status_words() {
  static StatusWords words;
  return words;
}

}  // namespace

struct zgr_ctx {
  int device = 0;
  int sm_count = 0;
  zgr_config cfg{};
  double a = 0, b = 0;
  int64_t d = 0, K = 0;
  std::vector<TensorDesc> descs;      // host mirror of the device table
  TensorDesc* d_descs = nullptr;
  bool descs_dirty = false;
  bool descs_fresh = false;           // copied to the device since the last sweep
  std::vector<void*> owned;           // device allocations made by the library
  std::vector<Group> groups;          // sweep plan
  // Small sets: the items of the CUDA-core contraction group with those of the isotropic group behind them, for one launch of the
  // contraction kernel instead of two (not while the kernels are timed or keep the norm bookkeeping, nor layer by layer).
  int merged_fma = -1, merged_iso = -1;
  WorkItem* d_merged = nullptr;
  std::vector<WorkItem> merged;
  std::vector<WorkItem> stats_items;  // plan of the norm kernel (tensors not served by the tcgen05 kernel)
  bool stats_planned = false;
  WorkItem* d_stats_items = nullptr;
  double* d_stats_slots = nullptr;    // slots of the separate norm pass over stats_items
  std::vector<int32_t> stats_first;   // per tensor: first item in stats_items (size n + 1)
  StatRange* d_ranges_pass = nullptr; // per tensor: where the separate pass leaves its partial sums
  StatRange* d_ranges_sweep = nullptr;  // per tensor: where a sweep with bookkeeping leaves them
  bool sweep_stats_ready = false;     // slots and ranges of the sweep plan exist
  bool stats_on = false;              // zgr_config.stats / zgr_enable_stats
  bool held_valid = false;            // the slots of the sweep plan hold the norms of held_seed, scaled by held_c^2
  uint64_t held_seed = 0;
  double held_c = 0.0;
  double* d_stats = nullptr;
  std::map<uint64_t, double> ledger;  // seeds whose perturbation is applied to the weights -> sum of the coefficients applied
  uint64_t last_seed = 0;             // most recently swept seed (introspection)
  bool guided_at_init = false;        // b != 0 when the sweep plan was made
  SplitJob* d_split_jobs = nullptr;   // one job per tensor served by a tcgen05 kernel: rebuild of its operand copies of U
  std::vector<SplitJob> split_jobs;   // the same on the host
  std::vector<int32_t> split_job;     // per tensor: its job, or -1
  int n_split_jobs = 0;
  std::vector<Group> groups_multi;    // plan of sweeps with several terms where it differs from `groups` (multi_groups)
  bool multi_planned = false;         // (of the legacy tensor-core path, on first use)
  int many_terms = 0;                 // from how many terms on (many_terms_from); 0: never
  int sticky = 0;                     // first CUDA failure, returned by every later call
  int64_t launches = 0;
  bool profiling = false;
  std::vector<int32_t> profiled;      // kernel_number of the entries of the last zgr_profile_read
  CUtensorMap* d_tmaps = nullptr;     // three per tensor (theta, U hi, U lo); tcgen05 path only
  std::vector<CUtensorMap> tmaps;     // host mirror
  int* d_err = nullptr;               // set by a kernel whose bounded wait gave up
  std::vector<cudaEvent_t> layer_events;  // zgr_perturb_layers: one per layer plus two, created on first use
  cudaStream_t aux_stream = nullptr;      // zgr_perturb_layers: odd layers run here, so that one layer's tail overlaps the next one's start
  void* d_qr = nullptr;               // scratch of zgr_build_subspace (grown on demand)
  size_t qr_bytes = 0;
  int* h_status = nullptr;            // host-mapped status word of zgr_build_subspace (see StatusWords)
  bool h_status_own = false;
};

namespace {

PhiloxKeys make_keys(uint64_t seed) {
  PhiloxKeys k;
  uint32_t k0 = static_cast<uint32_t>(seed), k1 = static_cast<uint32_t>(seed >> 32);
  for (int r = 0; r < 10; ++r) {
    k.k0[r] = k0;
    k.k1[r] = k1;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return k;
}

NormalScale make_scale(double s, int bits) {
  const double kTwoPi = 6.283185307179586476925286766559;
  const int nb = bits == 32 ? 23 : 16;
  const double off = std::ldexp(1.0, -(nb + 1)) - 1.0;
  NormalScale ns;
  ns.kr = static_cast<float>(-2.0 * std::log(2.0) * s * s);
  ns.s = static_cast<float>(s);
  ns.phase = static_cast<float>(kTwoPi * off + (s >= 0 ? -kTwoPi : -0.5 * kTwoPi));
  ns.u1_off = static_cast<float>(off);
  return ns;
}

// Power of two that brings the coefficient strips of the tcgen05 kernel near 1: the smallest k with
// cb 2^k >= 1/2, cb = sum_q |c_q| b (0 if there is no guided part in this call).
int kshift_for(double cb) {
  if (!(cb > 0.0) || !std::isfinite(cb)) return 0;
  const int k = static_cast<int>(std::ceil(-std::log2(cb))) - 1;
  return std::min(std::max(k, -24), 40);
}

using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                   const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// cuTensorMapEncodeTiled through the runtime (the library does not link against libcuda).
EncodeTiledFn encode_tiled_fn() {
  static EncodeTiledFn fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &q) == cudaSuccess && q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(ptr);
  }
  return fn;
}

// 2-D map over a row-major matrix of elements of `bytes` (2 or 4) bytes, rows `pitch` elements apart, box = box_cols x box_rows,
// swizzle matching the box's row length in bytes (32, 64 or 128).
bool make_map(CUtensorMap* out, const void* base, int bytes, int64_t rows, int64_t cols, int64_t pitch, int box_rows, int box_cols) {
  EncodeTiledFn fn = encode_tiled_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(rows)};
  const cuuint64_t strides[1] = {static_cast<cuuint64_t>(pitch * bytes)};
  const cuuint32_t box[2] = {static_cast<cuuint32_t>(box_cols), static_cast<cuuint32_t>(box_rows)};
  const cuuint32_t estr[2] = {1, 1};
  const int row_bytes = box_cols * bytes;
  const CUtensorMapSwizzle sw = row_bytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : (row_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
  return fn(out, bytes == 4 ? CU_TENSOR_MAP_DATA_TYPE_UINT32 : CU_TENSOR_MAP_DATA_TYPE_UINT16, 2, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
bool make_map_16bit(CUtensorMap* out, const void* base, int64_t rows, int64_t cols, int box_cols) {
  return make_map(out, base, 2, rows, cols, cols, 128, box_cols);
}
// Map over a part of U kept in the order of staged_copy_row whose boxes are 128 rows in their own order: a box takes 16 rows of each of a
// span's eight residues, residue by residue within a row of eight.
bool make_map_in_order(CUtensorMap* out, const void* base, int64_t rows_pad, int kpad) {
  EncodeTiledFn fn = encode_tiled_fn();
  if (!fn) return false;
  const cuuint64_t row = static_cast<cuuint64_t>(kpad) * 2;
  const cuuint64_t dims[4] = {static_cast<cuuint64_t>(kpad), 8, 32, static_cast<cuuint64_t>(rows_pad / 256)};
  const cuuint64_t strides[3] = {32 * row, row, 256 * row};
  const cuuint32_t box[4] = {static_cast<cuuint32_t>(kpad), 8, 16, 1};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  const CUtensorMapSwizzle sw = kpad == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : (kpad == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
  return fn(out, CU_TENSOR_MAP_DATA_TYPE_UINT16, 4, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, sw,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The maps of a tensor of sweep_staged_kernel: of its weights, one per residue of the row modulo 8 if the rows are no multiple of eight
// elements (see zgr_staged.cu), and behind them the three parts of U, rows_pad x kpad each.
int n_weight_maps(const TensorDesc& td) { return (td.cols & 7) ? 8 : 1; }
bool make_weight_maps(CUtensorMap* out, const TensorDesc& td, void* data, int bytes) {
  if ((td.cols & 7) == 0) return make_map(out, data, bytes, td.rows, td.cols, td.cols, 128, 128 / bytes);
  for (int64_t i = 0; i < 8 && i < td.rows; ++i) {      // (residues without rows have no boxes)
    const int64_t shift = -(i * td.cols) & 7;
    if (!make_map(out + i, static_cast<uint8_t*>(data) + (i * td.cols + shift) * bytes, bytes, (td.rows - i + 7) / 8, (td.cols - shift) & ~int64_t{7},
                  8 * td.cols, 32, 128 / bytes))
      return false;
  }
  return true;
}
// Rows of such a tensor that are no multiple of eight elements are worked on in the order of the copies of U (staged_copy_row): in spans of
// 256 rows, residues 0-3 and 4-7 of a span a block of 128 each.
bool by_residue(const TensorDesc& td) { return td.staged && (td.cols & 7); }
int64_t copy_rows(const TensorDesc& td) { return by_residue(td) ? (td.rows + 255) / 256 * 256 : (td.rows + 127) / 128 * 128; }
// Rows of the tensor in front of block `block` of that order.
int64_t rows_before(const TensorDesc& td, int64_t block) {
  const int64_t row0 = std::min(block / 2 * 256, td.rows), span = std::min<int64_t>(td.rows - row0, 256);
  return row0 + (block & 1 ? span / 8 * 4 + std::min<int64_t>(span & 7, 4) : 0);
}
// Blocks of a tensor of so many rows that hold any: residues 4-7 of the last span may be empty.
int64_t blocks_in_spans(int64_t rows) { return rows / 256 * 2 + ((rows & 255) > 4 ? 2 : (rows & 255) > 0); }
// First row and number of rows of an item: of the tensor, or, on the staged kernel, in that order.
std::pair<int64_t, int64_t> item_rows(const TensorDesc& td, const KernelChoice& kc, const WorkItem& w) {
  if (!kc.staged || !by_residue(td)) return {w.row0_or_e0, w.nrows_or_count};
  const int64_t first = rows_before(td, w.row0_or_e0 / 128);
  return {first, rows_before(td, (w.row0_or_e0 + w.nrows_or_count) / 128) - first};
}

bool whole_octets(const zgr_tensor& t) { return (reinterpret_cast<uintptr_t>(t.data) & 15) == 0 && (t.cols % 8 == 0); }
// Weights of a model by storage, of those kinds of tensors whose kernel depends on how many there are: rank <= 8 in whole octets, and
// all that the kernels with three-part operands may serve.
struct SetSizes {
  int64_t low[2] = {0, 0}, three_part[2] = {0, 0};      // [0] 16-bit, [1] fp32
  // of the latter those in whole octets, the tiles of 128 x 128 that they fill and the strips of these, and the tiles of ragged 16-bit rows on the tile
  // kernel and, in spans of 256 rows, on the staged one
  int64_t octets[2] = {0, 0}, octet_tiles[2] = {0, 0}, octet_strips[2] = {0, 0}, ragged_tiles[2] = {0, 0}, ragged_strips = 0;
};
SetSizes set_sizes(const zgr_tensor* tensors, int32_t n) {
  SetSizes s;
  for (int32_t l = 0; l < n; ++l) {
    const zgr_tensor& t = tensors[l];
    if (t.rank == 0) continue;
    const int f32 = t.dtype == ZGR_F32;
    const bool low = t.rank <= 8 && whole_octets(t);
    if (low) s.low[f32] += t.rows * t.cols;
    if (!low && !f32 && whole_octets(t)) continue;
    s.three_part[f32] += t.rows * t.cols;
    const int64_t strips = (t.cols + 127) / 128, tiles = (t.rows + 127) / 128 * strips;
    if (whole_octets(t)) {
      s.octets[f32] += t.rows * t.cols;
      s.octet_tiles[f32] += tiles;
      s.octet_strips[f32] += strips;
    } else if (!f32) {
      s.ragged_tiles[0] += tiles;
      s.ragged_tiles[1] += blocks_in_spans(t.rows) * strips;
      s.ragged_strips += strips;
    }
  }
  return s;
}
// Do the ragged 16-bit tensors of a set take less time on the staged kernel?  Its tile is shorter, the less so the more seeds share it, but spans
// of 256 rows may cost some more of them on the busiest SM: 8.04 tiles a mean against 7.97 are nine against eight in shares (18 M weights in
// rows of 1234 and 4937, tile kernel / staged: one seed 135 / 95 us, three 61.5 / 60.2, four 71.7 / 74.5, eight 123.5 / 131.8).
bool ragged_on_staged(const SetSizes& sizes, int sm_count, int n_terms) {
  const double tile = n_terms == 1 ? 0.75 : (n_terms == 2 ? 0.85 : (n_terms == 3 ? 0.88 : 0.94));
  const double on_tile = static_cast<double>(sizes.ragged_tiles[0]) / sm_count, on_staged = static_cast<double>(sizes.ragged_tiles[1]) / sm_count;
  return on_staged < 12.0 ? tile * std::ceil(on_staged) <= std::ceil(on_tile) : tile * on_staged <= on_tile;      // (dealt out whole in shares)
}

// Which kernel family serves a tensor: 1 the TMA-staged one with two-part operands (16-bit weights in whole octets, rank > 8), 2 those with
// three-part operands (everything else with a subspace), 0 neither.  Small sets of rank <= 8 stay with the CUDA-core kernel, which starts
// faster and cuts finer (a step of 2.0 M bf16 weights, rank 8: 25 us there; 4.0 M: 42, 28 on the tile kernel).
// Rank <= 8 takes no operand copies in two fp16 parts: those hold 22 bits of entries up to 2^16 2^-ushift, and the fp32
// multiply-adds of the CUDA-core kernel, which serves the same tensors in a smaller set, have neither limit (the TMA-staged kernel:
// 776 us at 300 M).
int tensor_core_kind(const zgr_tensor& t, bool guided_on, const SetSizes& sizes) {
  if (!guided_on || t.rank == 0 || t.rows >= (int64_t{1} << 31) - 256) return 0;
  const bool vec = whole_octets(t);
  if (vec && t.rank <= 8) {
    const int64_t set = sizes.low[t.dtype == ZGR_F32];
    if (set < (int64_t{1} << 21)) return 0;
    // (at rank 4 three quarters of the contraction are padding, and on fp32 sets that keep every SM busy for long the CUDA-core kernel catches up.
    // us a step on CUDA cores / staged, 16 random bits:  rank 4  24 M 154 / 136, 63 M 332 / 331, 126 M 629 / 635, 1.2 G 4333 / 4371;
    // rank 8  63 M 365 / 333, 126 M 681 / 640, 354 M 1796 / 1759; with 32 bits 101 M 616 / 573; ranks 2 and 3 were not timed and go with rank 4)
    // Rank 1 leaves at 2^25 already: its one multiply-add is exact to a rounding, 2.5e-8 against 2.95e-8 of the six products.
    if (t.dtype == ZGR_F32 && t.rank <= 4 && set >= (int64_t{1} << (t.rank == 1 ? 25 : 26))) return 0;
    return 2;
  }
  // (the TMA-staged kernel keeps the high counter word of the generator fixed: fewer than 2^32 blocks of four elements)
  if (vec && t.dtype != ZGR_F32 && t.rows * t.cols < (int64_t{1} << 34)) return t.cols < (int64_t{1} << 31) - 256 ? 1 : 0;
  return 2;
}

// Which of the two kernels with three-part operands: 1 the staged one, 0 the tile kernel.  TMA wants the weights on a 16-byte boundary
// and rows that hold a whole octet wherever it begins; the staged kernel keeps the high counter word of the generator fixed.
// Small sets stay with the tile kernel, whose sixteen epilogue warps share every tile (two groups on alternate tiles leave half of
// them idle when a CTA has one or two): us a step tile / staged, bf16 rank 8 2.4 M 26.8 / 29.6, 4.0 M 32.1 / 31.7, 8 M 59.8 / 57.5; ragged
// 16-bit rank 16 1.6 M 34.0 / 42.6, 2.7 M 47.0 / 45.5, 3.0 M 48.5 / 44.6, 18 M 135 / 95; fp32 up to rank 16 3.1 M 38.4 / 39.0, 5.9 M 58.1 / 59.7,
// 6.3 M 49.9 / 51.4, 7.1 M 49.2 / 48.8, 19 M 106 / 101; fp32 above rank 16 3.9 M 49.2 / 47.9, 4.9 M 57.2 / 54.3, 6.3 M 70.2 / 63.7.
// fp32 rows that are no multiple of eight elements do so at any size: 96 M weights of rank 16 in rows of 1001 and 4001 469 / 479 (the accurate
// transform hides what the tile kernel spends on its transposition, and the residues cost half-empty tiles).
//
// Tiles that are not full cost the staged kernel more (its groups take full and half-empty ones in turn), so whole octets stay with the tile
// kernel where less than 0.7 of the tiles' area is filled; in fp32 up to rank 16 only, there also below 0.83 in strips of under 3.5 tiles.  16-bit
// rank 8, matrices of d and 4 d, 40 or 20 layers: d = 136, .38 99 / 107; 192, .68 115 / 128; 320, .78 162 / 161; 448, .84 111 / 106.  fp32 rank 4 to 16:
// 168, .52 148 / 156; 200, .67 156 / 165; 320, .78 193 / 186; 337 x 1424, .81 153 / 154, and beside ragged tensors 592 / 612; 337 x 1408, .88
// 129 / 123; fp32 rank 64, 192, .68 207 / 190.
// So do 16-bit sets of many items (from the counter) in strips of under four tiles: d = 256, 2.7 146 / 152; 320, 3.8 253 / 264; 384, 4.0 141 / 132.
// Ragged rows: ragged_on_staged (d = 125, 20 tiles a layer against 12, 86 / 105; 261, 114 against 90, 191 / 171).
int staged_kind(const zgr_tensor& t, const SetSizes& sizes, int sm_count) {
  const int f32 = t.dtype == ZGR_F32;
  if ((reinterpret_cast<uintptr_t>(t.data) & 15) != 0 || t.cols < 16 || t.cols >= (int64_t{1} << 31) - 256 || t.rows * t.cols >= (int64_t{1} << 34)) return 0;
  if ((t.cols & 7) != 0) return !f32 && sizes.three_part[0] >= 5 * (int64_t{1} << 19) && ragged_on_staged(sizes, sm_count, 1);
  const double full = static_cast<double>(sizes.octets[f32]) / (16384.0 * static_cast<double>(sizes.octet_tiles[f32]));
  if (f32 && t.rank > 16) return sizes.three_part[1] >= 5 * (int64_t{1} << 19);
  if (f32) return sizes.three_part[1] >= 13 * (int64_t{1} << 19) && full >= (2 * sizes.octet_tiles[1] < 7 * sizes.octet_strips[1] ? 0.83 : 0.7);
  const bool short_items = sizes.octet_tiles[0] >= 12 * sm_count && sizes.octet_tiles[0] < 4 * sizes.octet_strips[0];
  return sizes.three_part[0] >= 5 * (int64_t{1} << 19) && full >= 0.7 && !short_items;
}

bool umma_wanted() {
  const char* e = std::getenv("ZGR_TENSOR_PATH");
  return !(e && std::strcmp(e, "legacy") == 0);
}

int blocks_per_sm(const KernelChoice& kc, bool multi = false, bool stats = false) {
  if (is_tile(kc)) return 1;
  switch (kc.path) {
    case PATH_ISO: return iso_blocks_per_sm(kc.precise != 0, multi, stats);
    case PATH_GENERIC: return 4;
    case PATH_UMMA: return 1;
    default: return 2;
  }
}

struct Member {
  int tensor, strip, row_step;
  int64_t rows;                                           // to be cut: the tensor's, or its blocks in the order of the copies of U
};

// Append the items of one tensor: strips of `strip` columns, each cut into even chunks of at most about nrows rows.
void cut_tensor(const TensorDesc& t, const Member& m, int64_t nrows_for_strip(int64_t, int), int64_t arg, std::vector<WorkItem>& items) {
  for (int64_t c0 = 0; c0 < t.cols; c0 += m.strip) {
    const int ncols = static_cast<int>(std::min<int64_t>(m.strip, t.cols - c0));
    int64_t nrows = std::max<int64_t>(1, nrows_for_strip(arg, ncols));
    nrows = ((nrows + m.row_step - 1) / m.row_step) * m.row_step;
    const int64_t n_chunks = (m.rows + nrows - 1) / nrows;
    nrows = (m.rows + n_chunks - 1) / n_chunks;
    nrows = ((nrows + m.row_step - 1) / m.row_step) * m.row_step;
    for (int64_t r0 = 0; r0 < m.rows; r0 += nrows) items.push_back(WorkItem{m.tensor, ncols, r0, std::min(nrows, m.rows - r0), c0});
  }
}

// Small sets on the tensor-core kernels: the strips, one after the other, are cut into one contiguous share per CTA, all shares
// costing the same (in units of a 128 x 128 tile: the tiles, `strip_cost` times the rank for every 128 columns of a strip
// begun, `item_cost` for every item begun).  A CTA then builds one or two strips instead of one per item.  Items begin at multiples of `step`
// rows.  Returns the cost of a share; if that is not below `limit` (0: none), nothing is written.
double share_out(const std::vector<TensorDesc>& descs, const std::vector<Member>& members, int strip_cols, int step, int sm_count, double strip_cost, double item_cost,
                 double limit, std::vector<WorkItem>& items, std::vector<int32_t>& starts) {
  const auto fill = [&](double share, bool emit) -> int {
    int cta = 0;
    double room = share;
    if (emit) starts.assign(1, 0);
    for (const Member& m : members) {
      const TensorDesc& t = descs[m.tensor];
      const int64_t blocks = (m.rows + step - 1) / step;
      for (int64_t c0 = 0; c0 < t.cols; c0 += strip_cols) {
        const int ncols = static_cast<int>(std::min<int64_t>(strip_cols, t.cols - c0));
        const double tiles = (ncols + 127) / 128, wide = tiles * static_cast<double>(step / 128), begin = strip_cost * t.rank * tiles + item_cost;
        for (int64_t at = 0, take; at < blocks; at += take) {
          if (room < begin + wide && room < share) {
            ++cta;
            room = share;
            if (emit) starts.push_back(static_cast<int32_t>(items.size()));
          }
          take = std::min<int64_t>(std::max<int64_t>(static_cast<int64_t>((room - begin) / wide + 1e-9), 1), blocks - at);
          room -= begin + wide * static_cast<double>(take);
          if (emit) items.push_back(WorkItem{m.tensor, ncols, step * at, std::min<int64_t>(step * take, m.rows - step * at), c0});
        }
      }
    }
    if (emit) starts.push_back(static_cast<int32_t>(items.size()));
    return cta + 1;
  };
  double tiles = 0.0;
  for (const Member& m : members) tiles += static_cast<double>((m.rows + 127) / 128 * ((descs[m.tensor].cols + 127) / 128));
  double low = tiles / sm_count, high = 1.25 * low + 1.0;     // (the tiles alone take `low`)
  if (limit > 0.0) {
    if (limit <= low || fill(limit, false) > sm_count) return limit;
    high = std::min(high, limit);
  }
  while (fill(high, false) > sm_count) {
    low = high;
    high *= 1.5;
  }
  for (int i = 0; i < 10; ++i) {
    const double mid = 0.5 * (low + high);
    (fill(mid, false) <= sm_count ? high : low) = mid;
  }
  if (limit > 0.0 && high >= limit) return limit;
  items.clear();
  fill(high, true);
  return high;
}

// Work items of one group.  An item is a strip of columns x a range of rows; it costs its tiles and, once, its coefficient
// strip, so few tall items are cheap but divide badly over the SMs.  `target`: elements per item for about 16 rounds.
// In shares below `shares_below` tiles per SM on the three-part kernels.
void plan_tiles(const std::vector<TensorDesc>& descs, const std::vector<Member>& members, int sm_count, int64_t target, int shares_below, Group& g) {
  const auto by_elements = [](int64_t elements, int ncols) { return elements / ncols; };
  const auto by_rows = [](int64_t rows, int) { return rows; };
  const bool tile = is_tile(g.kc);
  if (g.kc.path == PATH_FMA && !tile) {
    // handed out by a counter: nine items per CTA on large sets; down to as many rows as make the strip half of an item's
    // generator work when there is too little to go round
    int64_t total = 0;
    for (const Member& m : members) total += descs[m.tensor].rows * descs[m.tensor].cols;
    const int64_t least = std::min<int64_t>(256 * 2 * g.kc.kpad, 16384);
    const int64_t per = std::min<int64_t>(std::max<int64_t>(total / (static_cast<int64_t>(sm_count) * 2 * 8), least), 1048576);
    for (const Member& m : members) cut_tensor(descs[m.tensor], m, by_elements, per, g.items);
    return;
  }
  int64_t tiles = 0;
  for (const Member& m : members) tiles += ((descs[m.tensor].rows + 127) / 128) * ((descs[m.tensor].cols + 127) / 128);
  const int64_t sms = sm_count;
  if (tile ? tiles < shares_below * sms : g.kc.path == PATH_UMMA && tiles < 24 * sms) {
    // per 128 columns and rank about a hundredth of a tile for the strip, twice that for fp32 (anything from 1/60 to 1/200 gives the
    // same times); an item has a pipeline to fill, which the three-part kernels do ahead where two strips fit
    const double strip_cost = g.kc.precise ? 0.02 : 0.01;
    const double item_cost = tile && g.kc.kpad < 64 ? 0.3 : 0.7;
    const int widest = members.empty() ? 128 : members[0].strip, step = members.empty() ? 128 : members[0].row_step;      // (the same for all of a group)
    const double best = share_out(descs, members, widest, step, sm_count, strip_cost, item_cost, 0.0, g.items, g.starts);
    if (widest > 128) {
      std::vector<WorkItem> items;
      std::vector<int32_t> starts;
      if (share_out(descs, members, 128, step, sm_count, strip_cost, item_cost, 0.0, items, starts) < best) {
        g.items.swap(items);
        g.starts.swap(starts);
      }
    }
    // Halves of spans of 256 rows where there are more spans than SMs and the shares come out smaller by more than the search resolves: in
    // whole spans 18 M weights in rows of 1234 and 4937 are 119 shares for 148 SMs.
    if (step > 128 && tiles > 2 * sms) share_out(descs, members, widest, 128, sm_count, strip_cost, item_cost, 0.98 * best, g.items, g.starts);
    return;
  }
  if (!tile) {
    for (const Member& m : members)
      cut_tensor(descs[m.tensor], m, by_elements, g.kc.path == PATH_UMMA ? 2 * target : target, g.items);
    return;
  }
  // Handed out by a counter to one CTA per SM.  Tall items are cheap (an item costs its 128 x 128 tiles and, per 512 octets of
  // its strip, 0.2 to 0.6 of a tile: fp32 rank 32 took 451 us a sweep in items of one tile, 344 in items of eight), small ones
  // finish evenly: the height for the first two thirds of the work and that for the last third are those that the list
  // scheduling of the items, replayed here, ends with first.  Half of a last item is added, because the tiles do not take
  // equally long in fact (119 M bf16 weights in rows of 1234: 565 us a step with 8 and 8 tiles, 536 with 8 and 2).
  const double item_cost = 0.15 + (0.2 + 0.2 * g.kc.precise + (g.kc.precise && g.kc.bits == 32 ? 0.2 : 0.0)) * ((19 * g.kc.kpad + 511) / 512) +
                           (g.kc.kpad == 64 ? 0.3 : 0.0);
  double best = 0.0;
  const bool spans = !members.empty() && members[0].row_step == 256;      // (one step for all tensors of a group)
  const auto blocks_of = [&](int64_t rows) { return spans ? (rows + 255) / 256 * 2 : (rows + 127) / 128; };
  std::vector<WorkItem> trial;
  std::vector<double> free_at(static_cast<size_t>(sm_count));
  if (tiles >= 64 * sms) {
    // Long sweeps: even also when dealt out in turn, so that neither the model below nor the counter has to be right: eight tiles, or nine
    // where that is even and eight is not (rows of 50265).  Sets that neither deals evenly are replayed with both, in spans with eight.
    // us a step with 8 / 9 / 6 / 4 tiles: RoBERTa-shaped fp32 rank 8 1732 / 1722 / 1776 / 1778, 13 layers of 1024 822 / 824 / 839 / 830, fp32 rank 32
    // of 1152 1142 / 1157 / 1131 / 1170, 16-bit rank 8 of 2048 1200 / 1205 / 1245 / 1277: eight or nine makes no difference beyond 1 %, lower ones cost.
    for (int64_t height : {8, 9}) {
      if (spans && height == 9) continue;
      trial.clear();
      for (const Member& m : members) cut_tensor(descs[m.tensor], m, by_rows, 128 * height, trial);
      std::fill(free_at.begin(), free_at.end(), 0.0);
      double total = 0.0;
      size_t cta = 0;
      for (const WorkItem& w : trial) {
        const double weights = static_cast<double>(item_rows(descs[w.tensor], g.kc, w).second) * w.ncols;
        total += weights;
        free_at[cta] += weights;
        if (++cta == free_at.size()) cta = 0;
      }
      if (*std::max_element(free_at.begin(), free_at.end()) <= 1.025 * total / static_cast<double>(sm_count)) {
        g.items.swap(trial);
        return;
      }
    }
  }
  for (int64_t big : {16, 12, 8, 9, 6, 4, 3, 2, 1})
    for (int64_t small : {big, std::max<int64_t>(big / 4, 1)}) {
      if (tiles >= 64 * sms ? small != big || (big != 8 && big != 9) : big == 9) continue;
      if (spans && (big & 3) != 0 && big != 2) continue;      // (rows in spans of 256: nothing between two and four blocks, and six is left out)
      if (best > 0.0 && tiles < 64 * sms && (small == big ? tiles / big > 16 * sms : tiles / big > 10 * sms || big == 1)) continue;
      // No schedule ends before the mean load: heights that cannot win are not cut into items, nor replayed to their end (the
      // search is a fourth of the time that setting up such a set takes).
      const double last = 0.5 * (static_cast<double>(small) + item_cost);
      if (best > 0.0) {
        int64_t done = 0, n_items = 0;
        for (const Member& m : members) {
          const int64_t strips = (descs[m.tensor].cols + 127) / 128, blocks = blocks_of(m.rows), h = 3 * done < 2 * tiles ? big : small;
          const int64_t chunks = (m.rows + 128 * h - 1) / (128 * h), tall = (blocks + chunks - 1) / chunks;
          n_items += strips * ((blocks + tall - 1) / tall);
          done += blocks * strips;
        }
        const double load = static_cast<double>(tiles) + static_cast<double>(n_items) * item_cost;
        if (load / static_cast<double>(sm_count) * (1.0 - 1e-9) + last >= best) continue;
      }
      trial.clear();
      int64_t done = 0;
      for (const Member& m : members) {
        cut_tensor(descs[m.tensor], m, by_rows, 128 * (3 * done < 2 * tiles ? big : small), trial);
        done += ((descs[m.tensor].rows + 127) / 128) * ((descs[m.tensor].cols + 127) / 128);
      }
      std::fill(free_at.begin(), free_at.end(), 0.0);      // heap with the CTA that is free first at [0]
      double end = 0.0;
      for (const WorkItem& w : trial) {
        if (best > 0.0 && end + last >= best) break;
        const double at = free_at[0] + static_cast<double>(blocks_of(w.nrows_or_count)) + item_cost;
        size_t i = 0;
        for (size_t c; (c = 2 * i + 1) < free_at.size(); i = c) {
          if (c + 1 < free_at.size() && free_at[c + 1] < free_at[c]) ++c;
          if (free_at[c] >= at) break;
          free_at[i] = free_at[c];
        }
        free_at[i] = at;
        end = std::max(end, at);
      }
      end += last;
      if (best == 0.0 || end < best) {
        best = end;
        g.items = trial;
      }
    }
}

// What sweeps of many terms do with tensors kept by residue: as with one term; on the tile kernel all the same; in shares up to 24 tiles per SM.
enum Many { MANY_AS_ONE = 0, MANY_ON_TILE = 1, MANY_IN_SHARES = 2 };

// Split the tensors listed in `which` into work items, grouped by the kernel that serves them.
// The kernel family follows the tensor's own storage type (fp32 tensors take the accurate transform and
// an exact fp32 contraction); `kernel_dtype` >= 0 overrides only the type the kernel reads and writes,
// which lets the test hook run a 16-bit tensor's kernel family on an fp32 image.
void plan(const std::vector<TensorDesc>& descs, const std::vector<int>& which, bool guided_on, int bits, int sm_count,
          std::vector<Group>& out, int kernel_dtype = -1, bool multi = false, Many many = MANY_AS_ONE) {
  int64_t total = 0;
  for (int l : which) total += descs[l].rows * descs[l].cols;
  // elements per item: enough items for ~16 rounds over the resident CTAs, but large enough that the
  // coefficient strip of an item is a small fraction of its work
  int64_t target = total / (static_cast<int64_t>(sm_count) * 2 * 16);
  target = std::min<int64_t>(std::max<int64_t>(target, 16384), 524288);

  std::map<std::tuple<int, int, int, int, int, int>, size_t> index;  // (path, dtype, kpad, precise, staged, by_residue) -> group
  auto group_for = [&](int path, int real_dtype, int kpad, int staged = 0, int by_res = 0) -> Group& {
    const int precise = real_dtype == ZGR_F32 ? 1 : 0;
    const int dtype = kernel_dtype >= 0 ? kernel_dtype : real_dtype;
    auto key = std::make_tuple(path, dtype, kpad, precise, staged, by_res);
    auto it = index.find(key);
    if (it == index.end()) {
      index[key] = out.size();
      Group g;
      g.kc = KernelChoice{path, dtype, kpad, bits, precise, staged, by_res};
      out.push_back(std::move(g));
      return out.back();
    }
    return out[it->second];
  };

  std::vector<std::vector<Member>> members;   // per group: the tensors it serves with strips of columns
  for (int l : which) {
    const TensorDesc& t = descs[l];
    const bool aligned = (reinterpret_cast<uintptr_t>(t.data) & 15) == 0;
    const bool guided = guided_on && t.rank > 0;
    if (!guided) {
      Group& g = group_for(PATH_ISO, t.dtype, 0);
      const int64_t n = t.rows * t.cols;
      // about three items per resident CTA (handed out by a counter), the larger the better for the loads in flight: 405 M bf16
      // weights take 977 us in items of 8192 elements, 905 in 32768, 890 in 65536
      const int64_t chunk = std::min<int64_t>(std::max<int64_t>(total / (static_cast<int64_t>(sm_count) * 8 * 3) / 2048 * 2048, 2048), 65536);
      for (int64_t e0 = 0; e0 < n; e0 += chunk)
        g.items.push_back(WorkItem{l, aligned ? 1 : 0, e0, std::min(chunk, n - e0), 0});
      continue;
    }
    const bool vec = aligned && (t.cols % 8 == 0);
    int path, kpad, strip, row_step, staged = 0, by_res = 0;
    const bool umma_ok = t.umma && kernel_dtype < 0;
    const bool tile_ok = t.tile && (kernel_dtype < 0 || kernel_dtype == t.dtype);
    if (tile_ok) {
      // fp32 with rank > 8, rows that are not a multiple of eight elements, and low ranks: three-part operands.  (The test hook
      // that sweeps an fp32 image of a 16-bit tensor keeps the one-element-per-thread kernel below.)
      path = vec && t.rank <= 8 ? PATH_FMA : PATH_GENERIC; kpad = t.kpad; strip = kTileStripCols;
      by_res = many == MANY_ON_TILE && by_residue(t);
      staged = t.staged && !by_res;
      row_step = staged && by_residue(t) ? 256 : 128;
    } else if (!vec || (t.rank > 8 && !umma_ok && (t.Ufrag == nullptr || multi))) {
      // (the legacy tensor-core kernel applies one term per sweep; several terms take the fallback)
      path = PATH_GENERIC; kpad = 0; strip = 64; row_step = 1;
    } else if (t.rank <= 8 && !umma_ok) {
      path = PATH_FMA; kpad = t.rank <= 4 ? 4 : 8; strip = 256; row_step = 1;
    } else if (umma_ok) {
      path = PATH_UMMA; kpad = t.kpad; strip = umma_strip_cols(kpad); row_step = 128;
    } else {
      path = PATH_MMA; kpad = t.rank <= 16 ? 16 : (t.rank <= 32 ? 32 : 64);
      strip = mma_strip_cols(kpad); row_step = mma_rows_per_iter(kpad);
    }
    Group& g = group_for(path, t.dtype, kpad, staged, by_res);
    const size_t gi = static_cast<size_t>(&g - out.data());
    if (members.size() <= gi) members.resize(gi + 1);
    members[gi].push_back(Member{l, strip, row_step, staged && by_residue(t) ? 128 * blocks_in_spans(t.rows) : t.rows});
  }
  members.resize(out.size());
  for (size_t gi = 0; gi < out.size(); ++gi)
    if (out[gi].kc.path != PATH_ISO)
      plan_tiles(descs, members[gi], sm_count, target, many == MANY_IN_SHARES && !members[gi].empty() && members[gi][0].row_step == 256 ? 24 : 12, out[gi]);
  for (Group& g : out) {
    g.elements = 0;
    for (const WorkItem& w : g.items) g.elements += g.kc.path == PATH_ISO ? w.nrows_or_count : item_rows(descs[w.tensor], g.kc, w).second * w.ncols;
  }
  for (Group& g : out)
    g.grid = !g.starts.empty() ? static_cast<int>(g.starts.size()) - 1 : static_cast<int>(std::min<int64_t>(static_cast<int64_t>(g.items.size()), static_cast<int64_t>(sm_count) * blocks_per_sm(g.kc)));
  // tensors were visited in ascending order, so each tensor's items are contiguous within its group
  for (Group& g : out) {
    g.first_item.assign(descs.size() + 1, static_cast<int32_t>(g.items.size()));
    for (size_t i = g.items.size(); i-- > 0;) g.first_item[static_cast<size_t>(g.items[i].tensor)] = static_cast<int32_t>(i);
    for (size_t l = descs.size(); l-- > 0;)
      if (g.first_item[l] > g.first_item[l + 1]) g.first_item[l] = g.first_item[l + 1];   // tensors without items in this group
    // (after the two passes first_item is non-decreasing and [first_item[l], first_item[l+1]) are the items of tensor l)
  }
}

int check(zgr_ctx* ctx, cudaError_t e) {
  if (e == cudaSuccess) return ZGR_OK;
  const int code = (e == cudaErrorMemoryAllocation) ? ZGR_ENOMEM : ZGR_ECUDA;
  if (ctx && ctx->sticky == 0) ctx->sticky = code;
  return code;
}

template <typename T>
int dev_alloc(zgr_ctx* ctx, T** p, size_t count) {
  void* q = nullptr;
  const int rc = check(ctx, cudaMalloc(&q, std::max<size_t>(count, 1) * sizeof(T)));
  if (rc != ZGR_OK) return rc;
  ctx->owned.push_back(q);
  *p = static_cast<T*>(q);
  return ZGR_OK;
}

// Device tables of a context, one allocation and one copy for all of them (an allocation takes about 0.4 ms when it needs fresh
// pages).  The sources are read by copy(), so that tables may hold addresses that place() gave.
class Tables {
  struct Part {
    void** at;
    const void* src;      // null: zeros
    size_t offset, bytes;
  };
  std::vector<Part> parts_;
  size_t image_ = 0;
  uint8_t* base_ = nullptr;

 public:
  template <typename T>
  void add(T** p, const T* src, size_t count) {
    parts_.push_back(Part{reinterpret_cast<void**>(p), src, image_, count * sizeof(T)});
    image_ += (std::max<size_t>(count, 1) * sizeof(T) + 255) / 256 * 256;
  }
  void add(Group& g) {
    if (g.items.empty()) return;
    add(&g.d_items, g.items.data(), g.items.size());
    if (!g.starts.empty()) add(&g.d_starts, g.starts.data(), g.starts.size());
    if (g.kc.path == PATH_FMA || g.kc.path == PATH_ISO || is_tile(g.kc)) add(&g.d_sched, static_cast<const int32_t*>(nullptr), 2);
  }
  // `extra` bytes behind the tables are not copied to.
  int place(zgr_ctx* ctx, size_t extra, uint8_t** extra_at) {
    const int rc = dev_alloc(ctx, &base_, image_ + extra);
    if (rc != ZGR_OK) return rc;
    for (const Part& t : parts_) *t.at = base_ + t.offset;
    if (extra_at) *extra_at = base_ + image_;
    return ZGR_OK;
  }
  int copy(zgr_ctx* ctx) {
    std::vector<uint8_t> image(image_, 0);
    for (const Part& t : parts_)
      if (t.src != nullptr && t.bytes > 0) std::memcpy(image.data() + t.offset, t.src, t.bytes);
    const int rc = check(ctx, cudaMemcpy(base_, image.data(), image_, cudaMemcpyHostToDevice));
    // the copy is not ordered with launches on the caller's (possibly non-blocking) streams
    return rc == ZGR_OK ? check(ctx, cudaDeviceSynchronize()) : rc;
  }
};

int upload_groups(zgr_ctx* ctx, std::vector<Group>& groups) {
  Tables tables;
  for (Group& g : groups) tables.add(g);
  const int rc = tables.place(ctx, 0, nullptr);
  return rc == ZGR_OK ? tables.copy(ctx) : rc;
}

// Do tensors of one group share storage with tensors of the other?  (Kernels of different families run one after the other.)
bool share_storage(const std::vector<TensorDesc>& descs, const Group& f, const Group& g) {
  std::vector<std::pair<uintptr_t, uintptr_t>> range[2];
  for (size_t l = 0; l < descs.size(); ++l)
    for (int i = 0; i < 2; ++i) {
      const Group& in = i == 0 ? f : g;
      const uintptr_t at = reinterpret_cast<uintptr_t>(descs[l].data);
      if (in.first_item[l + 1] > in.first_item[l]) range[i].emplace_back(at, at + static_cast<uintptr_t>(descs[l].rows * descs[l].cols * dtype_bytes(descs[l].dtype)));
    }
  std::sort(range[0].begin(), range[0].end());
  std::sort(range[1].begin(), range[1].end());
  uintptr_t reach[2] = {0, 0};               // end of the ranges that begin before the current one
  for (size_t i = 0, j = 0; i < range[0].size() || j < range[1].size();) {
    const int side = j == range[1].size() || (i < range[0].size() && range[0][i] < range[1][j]) ? 0 : 1;
    const auto& r = side == 0 ? range[0][i++] : range[1][j++];
    if (r.first < reach[1 - side]) return true;
    reach[side] = std::max(reach[side], r.second);
  }
  return false;
}

// The isotropic families go first: they are a few microseconds as a rule, during which the CTAs of the next kernel set up and make
// their first strip.  (Families that share storage with a matrix keep their place.)
void order_groups(const std::vector<TensorDesc>& descs, std::vector<Group>& groups) {
  for (size_t i = 1; i < groups.size(); ++i)
    for (size_t j = i; j > 0 && groups[j].kc.path == PATH_ISO && groups[j - 1].kc.path != PATH_ISO && !share_storage(descs, groups[j - 1], groups[j]); --j)
      std::swap(groups[j - 1], groups[j]);
}

// The isotropic elements that may ride along: up to 2^20, a few microseconds of one launch.
void merge_small_groups(zgr_ctx* ctx) {
  for (size_t i = 0; i < ctx->groups.size(); ++i)
    for (size_t j = 0; j < ctx->groups.size(); ++j) {
      const Group &f = ctx->groups[i], &g = ctx->groups[j];
      if (f.kc.path != PATH_FMA || is_tile(f.kc) || g.kc.path != PATH_ISO || f.kc.dtype != g.kc.dtype || f.kc.precise != g.kc.precise || g.items.empty() ||
          f.items.empty() || g.elements > (1 << 20) || share_storage(ctx->descs, f, g))
        continue;
      ctx->merged = f.items;
      ctx->merged.insert(ctx->merged.end(), g.items.begin(), g.items.end());
      ctx->merged_fma = static_cast<int>(i);
      ctx->merged_iso = static_cast<int>(j);
      return;
    }
}

// One sweep  theta <- rnd(theta + sum_q c_q z(seed_q))  over the planned groups (n terms, 1 <= n <= kMaxTerms).
// t0 <= t1 restricts the sweep to the tensors [t0, t1) (layer-wise sweeps); t1 < 0 means all of them.  tmaps: the tensor
// maps of the first tensor of d_descs (null: the context's own).
int sweep(zgr_ctx* ctx, std::vector<Group>& groups, const TensorDesc* d_descs, int n, const uint64_t* seeds, const double* c, cudaStream_t st,
          int32_t t0 = 0, int32_t t1 = -1, bool keep_stats = false, const CUtensorMap* tmaps = nullptr) {
  if (tmaps == nullptr) tmaps = ctx->d_tmaps;
  SweepParams p;
  std::memset(&p, 0, sizeof(p));
  for (int q = 0; q < n; ++q) {
    p.term[q].keys = make_keys(seeds[q]);
    p.term[q].iso = make_scale(c[q] * ctx->a, ctx->cfg.bits_per_normal);
    p.term[q].cb = static_cast<float>(c[q] * ctx->b);
  }
  p.n_terms = n;
  p.unit = make_scale(1.0, ctx->cfg.bits_per_normal);
  p.tensors = d_descs;
  double cb_total = 0.0;
  for (int q = 0; q < n; ++q) cb_total += std::fabs(c[q] * ctx->b);
  p.kshift = kshift_for(cb_total);
  const bool merge = ctx->d_merged != nullptr && &groups == &ctx->groups && !ctx->profiling && t1 < 0 && !keep_stats;
  const auto has_work = [&](const Group& g) {
    if (g.items.empty() || (merge && &g - groups.data() == ctx->merged_iso)) return false;
    return t1 < 0 || g.first_item[static_cast<size_t>(t1)] > g.first_item[static_cast<size_t>(t0)];
  };
  const Group* last = nullptr;
  for (const Group& g : groups)
    if (has_work(g)) last = &g;
  const bool early = !ctx->descs_fresh;      // (the kernels read the tensor table before they wait)
  ctx->descs_fresh = false;
  for (Group& g : groups) {
    if (!has_work(g)) continue;
    const int index = static_cast<int>(&g - groups.data());
    p.items = g.d_items;
    p.n_items = static_cast<int32_t>(g.items.size());
    p.item_stats = keep_stats ? g.d_item_stats : nullptr;
    p.item_base = 0;
    if (merge && index == ctx->merged_fma) {
      p.items = ctx->d_merged;
      p.n_items = static_cast<int32_t>(ctx->merged.size());
    }
    p.sched = g.d_sched ? g.d_sched + (ctx->aux_stream != nullptr && st == ctx->aux_stream ? 1 : 0) : nullptr;
    if (t1 >= 0) {
      const int32_t b0 = g.first_item[static_cast<size_t>(t0)], b1 = g.first_item[static_cast<size_t>(t1)];
      p.items = g.d_items + b0;
      p.n_items = b1 - b0;
      p.item_base = b0;
    }
    p.starts = t1 >= 0 ? nullptr : g.d_starts;
    const int grid = p.starts ? g.grid
                              : static_cast<int>(std::min<int64_t>(p.n_items, static_cast<int64_t>(ctx->sm_count) * blocks_per_sm(g.kc, n > 1, p.item_stats != nullptr)));
    p.early = early && &g != last ? 1 : 0;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (ctx->profiling && t1 < 0) {
      if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
        if (e0) cudaEventDestroy(e0);
        return check(ctx, cudaErrorUnknown);
      }
      cudaEventRecord(e0, st);
    }
    const int rc = check(ctx, g.kc.path == PATH_UMMA ? launch_sweep_umma(g.kc, p, tmaps, ctx->d_err, grid, st)
                              : g.kc.staged ? launch_sweep_staged(g.kc, p, ctx->d_err, grid, st)
                              : is_tile(g.kc) ? launch_sweep_tile(g.kc, p, tmaps, ctx->d_err, grid, st)
                                              : launch_sweep(g.kc, p, grid, st));
    if (rc != ZGR_OK) {
      if (e0) cudaEventDestroy(e0);
      if (e1) cudaEventDestroy(e1);
      return rc;
    }
    if (e0) {
      cudaEventRecord(e1, st);
      g.timed.emplace_back(e0, e1);
    }
    ctx->launches++;
  }
  return ZGR_OK;
}

int flush_descs(zgr_ctx* ctx, cudaStream_t st) {
  if (!ctx->descs_dirty) return ZGR_OK;
  const int rc = check(ctx, cudaMemcpyAsync(ctx->d_descs, ctx->descs.data(), ctx->descs.size() * sizeof(TensorDesc), cudaMemcpyHostToDevice, st));
  if (rc == ZGR_OK) {
    ctx->descs_dirty = false;
    ctx->descs_fresh = true;
  }
  return rc;
}

bool is_finite(double x) { return std::isfinite(x); }

// Fragment-order copy of U for the mma.sync kernel (made on demand for tensors that the tcgen05 kernel sweeps: only the test
// hook zgr_debug_z reads it there).
int make_fragments(zgr_ctx* ctx, TensorDesc& td, cudaStream_t st) {
  int rc = ZGR_OK;
  if (td.Ufrag == nullptr) {
    const size_t n_frag = static_cast<size_t>((td.rows + 15) / 16) * (td.kpad / 16) * 2 * 32;
    uint4* frag = nullptr;
    rc = dev_alloc(ctx, &frag, n_frag);
    if (rc != ZGR_OK) return rc;
    td.Ufrag = frag;
  }
  rc = check(ctx, launch_split_subspace(td.U, td.rows, td.rank, td.kpad, const_cast<uint4*>(td.Ufrag), st));
  if (rc == ZGR_OK) ctx->launches++;
  return rc;
}

// The jobs [first, first + count) of the operand copies, in one launch.
int split_jobs(zgr_ctx* ctx, int first, int count, cudaStream_t st) {
  int64_t most = 0;
  for (int i = first; i < first + count; ++i) most = std::max(most, ctx->split_jobs[static_cast<size_t>(i)].rows_pad * ctx->split_jobs[static_cast<size_t>(i)].kp);
  const int rc = check(ctx, launch_split_subspaces(ctx->d_split_jobs + first, count, most, st));
  if (rc == ZGR_OK && count > 0) ctx->launches++;
  return rc;
}

// Rebuild the library's operand copies of U for one tensor from the subspace buffer (enqueued on st).
int refresh_operands(zgr_ctx* ctx, int32_t tensor, cudaStream_t st) {
  TensorDesc& td = ctx->descs[static_cast<size_t>(tensor)];
  int rc = ZGR_OK;
  // (for a tensor of the tcgen05 kernel the fragment-order copy is only read by zgr_debug_z, which rebuilds it)
  if (td.Ufrag != nullptr && !td.umma) rc = make_fragments(ctx, td, st);
  const int32_t job = ctx->split_job[static_cast<size_t>(tensor)];
  if (rc == ZGR_OK && job >= 0) rc = split_jobs(ctx, job, 1, st);
  return rc;
}

// Bookkeeping slots of a plan: kStatSlots x 3 doubles per work item, zeroed once (slots that no warp owns stay
// zero; the others are rewritten by every launch that keeps the bookkeeping).
int alloc_slots(zgr_ctx* ctx, double** out, size_t n_items) {
  const size_t count = std::max<size_t>(n_items, 1) * kStatSlots * 3;
  int rc = dev_alloc(ctx, out, count);
  if (rc == ZGR_OK) rc = check(ctx, cudaMemset(*out, 0, count * sizeof(double)));
  return rc;
}

// In-sweep bookkeeping needs every group of the sweep plan to be a kernel family that keeps it.
bool sweep_stats_possible(const zgr_ctx* ctx) {
  for (const Group& g : ctx->groups)
    if (!g.items.empty() && g.kc.path == PATH_MMA) return false;
  return true;
}

int prepare_sweep_stats(zgr_ctx* ctx) {
  if (ctx->sweep_stats_ready) return ZGR_OK;
  const size_t n = ctx->descs.size();
  std::vector<StatRange> ranges(n, StatRange{nullptr, 0, 0});
  for (Group& g : ctx->groups) {
    if (g.items.empty()) continue;
    const int rc = alloc_slots(ctx, &g.d_item_stats, g.items.size());
    if (rc != ZGR_OK) return rc;
    for (size_t l = 0; l < n; ++l)
      if (g.first_item[l + 1] > g.first_item[l]) ranges[l] = StatRange{g.d_item_stats, g.first_item[l], g.first_item[l + 1] - g.first_item[l]};
  }
  int rc = dev_alloc(ctx, &ctx->d_ranges_sweep, n);
  if (rc == ZGR_OK) rc = check(ctx, cudaMemcpy(ctx->d_ranges_sweep, ranges.data(), n * sizeof(StatRange), cudaMemcpyHostToDevice));
  if (rc == ZGR_OK) ctx->sweep_stats_ready = true;
  return rc;
}

// A context's tables, tensor maps and borrowed pointers live on the device that was current at zgr_init.
// Launching from another current device would hand its kernels foreign addresses, so every entry point
// that enqueues work checks this first and refuses before anything is launched.
bool on_ctx_device(const zgr_ctx* ctx) {
  int cur = -1;
  if (cudaGetDevice(&cur) != cudaSuccess) return false;
  return zgr_debug_check_device(ctx->device, cur) == ZGR_OK;
}

// Mixing scalars of Eq. (perturbation) with n := d and m := K
void set_mixing(zgr_ctx* ctx, double alpha) {
  const double d = static_cast<double>(ctx->d), K = static_cast<double>(ctx->K);
  ctx->cfg.alpha = alpha;
  ctx->a = std::sqrt(alpha / d);
  ctx->b = ctx->K > 0 ? std::sqrt((1.0 - alpha) / K) : 0.0;
  if (ctx->cfg.scale_mode == ZGR_SCALE_UNIT) {
    ctx->a *= std::sqrt(d);
    ctx->b *= std::sqrt(d);
  }
}

// Argument checks shared by zgr_init and zgr_debug_plan; d = parameters, K = guided coefficients.
int validate_model(const zgr_tensor* tensors, int32_t n, const zgr_config* cfg, int64_t* d_out, int64_t* K_out) {
  if (!tensors || !cfg || n <= 0) return ZGR_EINVAL;
  if (!(cfg->alpha >= 0.0 && cfg->alpha <= 1.0) || !is_finite(cfg->eps) || !(cfg->eps > 0.0)) return ZGR_EINVAL;
  if (cfg->scale_mode != ZGR_SCALE_PAPER && cfg->scale_mode != ZGR_SCALE_UNIT) return ZGR_EINVAL;
  if (cfg->bits_per_normal != 32 && cfg->bits_per_normal != 16) return ZGR_EINVAL;
  int64_t d = 0, K = 0;
  for (int32_t l = 0; l < n; ++l) {
    const zgr_tensor& t = tensors[l];
    if (!t.data || t.rows < 1 || t.cols < 1) return ZGR_EINVAL;
    if (t.dtype != ZGR_F32 && t.dtype != ZGR_F16 && t.dtype != ZGR_BF16) return ZGR_EINVAL;
    if (t.rank < 0 || t.rank > ZGR_MAX_RANK) return ZGR_EINVAL;
    if ((t.rank == 0) != (t.U == nullptr)) return ZGR_EINVAL;
    if (reinterpret_cast<uintptr_t>(t.data) % dtype_bytes(t.dtype) != 0) return ZGR_EINVAL;
    if (t.U && reinterpret_cast<uintptr_t>(t.U) % 4 != 0) return ZGR_EINVAL;
    if (t.rows > (INT64_MAX / t.cols)) return ZGR_EINVAL;
    d += t.rows * t.cols;
    K += static_cast<int64_t>(t.rank) * t.cols;
  }
  *d_out = d;
  *K_out = K;
  return ZGR_OK;
}

// From how many terms on a sweep treats the set's ragged 16-bit tensors otherwise than single seeds, which the staged kernel serves, and how; 0:
// never.  Either on the tile kernel, or, where items from the counter are few and tall, in shares: they need not be cut as low as for one seed,
// whose layer-wise sweeps share the items out again, and the hand-out of tiles that many terms make long ends unevenly (us a pass from the
// counter / in shares: 64 M weights in rows of 1411 four seeds 212 / 182, eight of rank 40 399 / 334; 36 M of 999 rank 48 three seeds 130 / 108;
// 39 M of 683 eight 249 / 242; but strips of four tiles, 35 M of 384 at rank 8, four seeds 114 / 118).
int many_terms_from(const std::vector<TensorDesc>& descs, const SetSizes& sizes, int sm_count, Many* many) {
  bool ragged = false;
  for (const TensorDesc& td : descs) ragged = ragged || by_residue(td);
  *many = MANY_ON_TILE;
  for (int n = 2; ragged && n <= 4; ++n)
    if (!ragged_on_staged(sizes, sm_count, n)) return n;
  *many = MANY_IN_SHARES;
  const int64_t tiles = sizes.ragged_tiles[1];
  if (ragged && tiles >= 12 * sm_count && tiles < 24 * sm_count && tiles >= 6 * sizes.ragged_strips) return 2;
  *many = MANY_AS_ONE;
  return 0;
}

// The plan of a sweep as zgr_init would make it, without a device.
int plan_on_host(const zgr_tensor* tensors, int32_t n, const zgr_config* cfg, int sm_count, bool tcgen05, bool multi, std::vector<TensorDesc>& descs,
                 std::vector<Group>& groups) {
  int64_t d = 0, K = 0;
  const int valid = validate_model(tensors, n, cfg, &d, &K);
  if (valid != ZGR_OK) return valid;
  const bool guided_on = K > 0 && cfg->alpha < 1.0;
  const SetSizes sizes = set_sizes(tensors, n);
  descs.resize(static_cast<size_t>(n));
  std::vector<int> all(static_cast<size_t>(n));
  for (int32_t l = 0; l < n; ++l) {
    const zgr_tensor& t = tensors[l];
    TensorDesc& td = descs[static_cast<size_t>(l)];
    std::memset(&td, 0, sizeof(td));
    td.data = t.data; td.U = t.U; td.rows = t.rows; td.cols = t.cols; td.rank = t.rank; td.id = l; td.dtype = t.dtype; td.qbits = 8;
    const bool vec = (reinterpret_cast<uintptr_t>(t.data) & 15) == 0 && (t.cols % 8 == 0);
    if (guided_on && t.rank > 8 && vec && t.dtype != ZGR_F32) {
      // what zgr_init would have built for this tensor: operand copies for the tensor-core kernels
      td.kpad = t.rank <= 16 ? 16 : (t.rank <= 32 ? 32 : 64);
      td.Ufrag = reinterpret_cast<const uint4*>(uintptr_t{16});   // marker only: never dereferenced by the planner
    }
    const int kind = tcgen05 ? tensor_core_kind(t, guided_on, sizes) : 0;
    if (kind != 0) {
      td.kpad = t.rank <= 16 ? 16 : (t.rank <= 32 ? 32 : 64);
      (kind == 1 ? td.umma : td.tile) = 1;
      if (kind == 2) td.staged = staged_kind(t, sizes, sm_count);
    }
    all[static_cast<size_t>(l)] = l;
  }
  Many many = MANY_AS_ONE;
  if (multi) many_terms_from(descs, sizes, sm_count, &many);
  plan(descs, all, guided_on, cfg->bits_per_normal, sm_count, groups, -1, multi, many);
  return ZGR_OK;
}

// Book-keeping of the coefficients applied under each seed; a seed whose coefficients cancel is idle again.
void ledger_add(zgr_ctx* ctx, uint64_t seed, double c) {
  double& net = ctx->ledger[seed];
  net += c;
  if (net == 0.0) ctx->ledger.erase(seed);
  ctx->last_seed = seed;
}

// Plan used by sweeps with n terms, n > 1: the sweep plan itself unless it contains the legacy
// tensor-core kernel, which applies one term per sweep (those tensors are re-planned onto the fallback), or so many terms
// have a plan of their own.
std::vector<Group>& multi_groups(zgr_ctx* ctx, int n, int* rc) {
  *rc = ZGR_OK;
  if (ctx->many_terms > 0 && n >= ctx->many_terms) return ctx->groups_multi;
  bool legacy = false;
  for (const Group& g : ctx->groups) legacy = legacy || (g.kc.path == PATH_MMA && !g.items.empty());
  if (!legacy) return ctx->groups;
  if (!ctx->multi_planned) {
    std::vector<int> all(ctx->descs.size());
    for (size_t l = 0; l < all.size(); ++l) all[l] = static_cast<int>(l);
    plan(ctx->descs, all, ctx->guided_at_init, ctx->cfg.bits_per_normal, ctx->sm_count, ctx->groups_multi, -1, true);
    *rc = upload_groups(ctx, ctx->groups_multi);
    ctx->multi_planned = true;
  }
  return ctx->groups_multi;
}

}  // namespace

namespace zgr {
PhiloxKeys host_make_keys(uint64_t seed) { return make_keys(seed); }
NormalScale host_make_scale(double s, int bits) { return make_scale(s, bits); }
bool host_ctx_view(const zgr_ctx* ctx, int32_t l, TensorDesc* desc, double* a, double* b, int* bits, int* sticky, int* device) {
  if (!ctx || l < 0 || l >= static_cast<int32_t>(ctx->descs.size())) return false;
  *desc = ctx->descs[static_cast<size_t>(l)];
  *a = ctx->a;
  *b = ctx->b;
  *bits = ctx->cfg.bits_per_normal;
  *sticky = ctx->sticky;
  *device = ctx->device;
  return true;
}
}  // namespace zgr

// ------------------------------------------------------------------------------------------------
extern "C" {

int zgr_init(zgr_ctx** out, const zgr_tensor* tensors, int32_t n, const zgr_config* cfg) {
  if (!out) return ZGR_EINVAL;
  *out = nullptr;
  int64_t d = 0, K = 0;
  const int valid = validate_model(tensors, n, cfg, &d, &K);
  if (valid != ZGR_OK) return valid;

  zgr_ctx* ctx = new (std::nothrow) zgr_ctx();
  if (!ctx) return ZGR_ENOMEM;
  ctx->cfg = *cfg;
  ctx->stats_on = cfg->stats != 0;
  ctx->d = d;
  ctx->K = K;
  set_mixing(ctx, cfg->alpha);

  int rc = check(ctx, cudaGetDevice(&ctx->device));
  if (rc == ZGR_OK) rc = check(ctx, cudaDeviceGetAttribute(&ctx->sm_count, cudaDevAttrMultiProcessorCount, ctx->device));
  if (rc != ZGR_OK) {
    delete ctx;
    return rc;
  }

  ctx->descs.resize(static_cast<size_t>(n));
  ctx->tmaps.resize(static_cast<size_t>(3 * n));
  std::memset(ctx->tmaps.data(), 0, ctx->tmaps.size() * sizeof(CUtensorMap));
  const bool guided_on = ctx->b != 0.0;
  ctx->guided_at_init = guided_on;
  const SetSizes sizes = set_sizes(tensors, n);
  size_t operand_bytes = 0, n_staged_maps = 0;
  for (int32_t l = 0; l < n && rc == ZGR_OK; ++l) {
    const zgr_tensor& t = tensors[l];
    TensorDesc& td = ctx->descs[static_cast<size_t>(l)];
    td.data = t.data;
    td.U = t.U;
    td.Ufrag = nullptr;
    td.q = nullptr;
    td.qscale = nullptr;
    td.qzero = nullptr;
    td.qbits = 8;
    td.qrows = 0;
    td.rows = t.rows;
    td.cols = t.cols;
    td.rank = t.rank;
    td.kpad = 0;
    td.id = l;
    td.dtype = t.dtype;
    td.umma = 0;
    td.tile = 0;
    td.staged = 0;
    td.maps = nullptr;
    td.ushift = 0;
    for (void*& copy : td.Ucopy) copy = nullptr;
    // tcgen05 kernels: row-major copies of U in parts, and three tensor maps (those of the copies once these have their place)
    const int kind = umma_wanted() && encode_tiled_fn() != nullptr ? tensor_core_kind(t, guided_on, sizes) : 0;
    if (kind == 2 || (kind == 1 && make_map_16bit(&ctx->tmaps[static_cast<size_t>(3 * l)], t.data, t.rows, t.cols, 64))) {
      td.kpad = t.rank <= 16 ? 16 : (t.rank <= 32 ? 32 : 64);
      // entries of an orthonormal U are about 1/sqrt(rows): scaled by 2^ushift they sit between 1 and 2 in size
      // (capped at 2^12, which leaves fp16 room for entries up to 16 in size); the bf16 parts need no scaling
      if (kind == 1) td.ushift = std::min<int32_t>(12, static_cast<int32_t>(std::ceil(0.5 * std::log2(static_cast<double>(t.rows)))));
      (kind == 1 ? td.umma : td.tile) = 1;
      if (kind == 2) td.staged = staged_kind(t, sizes, ctx->sm_count);
      operand_bytes += (kind == 1 ? 2 : 3) * static_cast<size_t>(copy_rows(td)) * static_cast<size_t>(td.kpad) * 2;
      if (td.staged) n_staged_maps += static_cast<size_t>(n_weight_maps(td)) + 3;
    }
    const bool vec = (reinterpret_cast<uintptr_t>(t.data) & 15) == 0 && (t.cols % 8 == 0);
    if (guided_on && t.rank > 8 && vec && t.dtype != ZGR_F32 && !td.umma) {
      // the mma.sync kernel serves this tensor: copy of U in A-fragment order
      td.kpad = t.rank <= 16 ? 16 : (t.rank <= 32 ? 32 : 64);
      rc = make_fragments(ctx, td, nullptr);
    }
  }
  ctx->split_job.assign(static_cast<size_t>(n), -1);
  if (rc == ZGR_OK) {
    std::vector<SplitJob>& jobs = ctx->split_jobs;
    for (int32_t l = 0; l < n; ++l)
      if (ctx->descs[static_cast<size_t>(l)].umma || ctx->descs[static_cast<size_t>(l)].tile) ctx->split_job[static_cast<size_t>(l)] = ctx->n_split_jobs++;
    jobs.resize(static_cast<size_t>(ctx->n_split_jobs));
    std::vector<int> all(static_cast<size_t>(n));
    for (int32_t l = 0; l < n; ++l) all[static_cast<size_t>(l)] = l;
    plan(ctx->descs, all, guided_on, cfg->bits_per_normal, ctx->sm_count, ctx->groups);
    order_groups(ctx->descs, ctx->groups);
    merge_small_groups(ctx);
    Many many;
    ctx->many_terms = many_terms_from(ctx->descs, sizes, ctx->sm_count, &many);
    if (ctx->many_terms > 0) {
      plan(ctx->descs, all, guided_on, cfg->bits_per_normal, ctx->sm_count, ctx->groups_multi, -1, true, many);
      order_groups(ctx->descs, ctx->groups_multi);
    }
    Tables tables;
    tables.add(&ctx->d_split_jobs, jobs.data(), jobs.size());
    std::vector<CUtensorMap> staged_maps(n_staged_maps);
    CUtensorMap* d_staged_maps = nullptr;
    tables.add(&ctx->d_tmaps, ctx->tmaps.data(), ctx->tmaps.size());
    tables.add(&d_staged_maps, staged_maps.data(), staged_maps.size());
    tables.add(&ctx->d_descs, ctx->descs.data(), ctx->descs.size());
    tables.add(&ctx->d_err, static_cast<const int*>(nullptr), 1);
    tables.add(&ctx->d_stats, static_cast<const double*>(nullptr), static_cast<size_t>(3 * n));
    for (Group& g : ctx->groups) tables.add(g);
    for (Group& g : ctx->groups_multi) tables.add(g);
    if (!ctx->merged.empty()) tables.add(&ctx->d_merged, ctx->merged.data(), ctx->merged.size());
    // Scratch of zgr_build_subspace, up to 2 MB (every rank up to 32, and rank 64 in one cluster): as an allocation of its own inside the
    // first call it would be most of that call.  Its first 512 bytes are the last of the zeroed tables.
    size_t scratch = 0;
    for (int32_t l = 0; l < n; ++l) {
      const zgr_tensor& t = tensors[l];
      if (t.rank == 0 || t.rows < t.rank || !subspace_fused(t.rows, t.rank, ctx->sm_count)) continue;
      const size_t need = subspace_scratch_bytes(t.rows, t.rank, ctx->sm_count);
      if (need <= (size_t{2} << 20)) scratch = std::max(scratch, need);
    }
    uint8_t *at = nullptr, *qr = nullptr;
    if (scratch > 0) tables.add(&qr, static_cast<const uint8_t*>(nullptr), 512);
    const size_t behind = scratch > 0 ? (scratch - 512 + 255) / 256 * 256 : 0;
    rc = tables.place(ctx, behind + operand_bytes, &at);
    if (rc == ZGR_OK) {
      at += behind;
      ctx->d_qr = qr;
      ctx->qr_bytes = scratch;
    }
    size_t map_at = 0;
    for (int32_t l = 0; l < n && rc == ZGR_OK; ++l) {
      TensorDesc& td = ctx->descs[static_cast<size_t>(l)];
      const int32_t job = ctx->split_job[static_cast<size_t>(l)];
      if (job < 0) continue;
      const int64_t rows_pad = copy_rows(td);
      CUtensorMap* m = &ctx->tmaps[static_cast<size_t>(3 * l)] + (td.umma ? 1 : 0);
      if (td.staged) {
        td.maps = d_staged_maps + map_at;
        m = &staged_maps[map_at];
        if (!make_weight_maps(m, td, td.data, dtype_bytes(td.dtype))) rc = check(ctx, cudaErrorUnknown);
        m += n_weight_maps(td);
        map_at += static_cast<size_t>(n_weight_maps(td)) + 3;
      }
      for (int i = 0; i < (td.umma ? 2 : 3); ++i) {
        td.Ucopy[i] = at;
        if (!make_map_16bit(m + i, at, rows_pad, td.kpad, td.kpad)) rc = check(ctx, cudaErrorUnknown);
        if (many == MANY_ON_TILE && by_residue(td) && !make_map_in_order(&ctx->tmaps[static_cast<size_t>(3 * l + i)], at, rows_pad, td.kpad))
          rc = check(ctx, cudaErrorUnknown);
        at += static_cast<size_t>(rows_pad) * td.kpad * 2;       // (a multiple of 4096 bytes)
      }
      jobs[static_cast<size_t>(job)] = SplitJob{td.U, {td.Ucopy[0], td.Ucopy[1], td.Ucopy[2]}, td.rows, rows_pad, td.rank, td.kpad, td.umma ? td.ushift : -1,
                                                  by_residue(td) ? 1 : 0};
    }
    if (rc == ZGR_OK) rc = tables.copy(ctx);
    if (rc == ZGR_OK) rc = split_jobs(ctx, 0, ctx->n_split_jobs, nullptr);
  }
  if (rc == ZGR_OK) rc = check(ctx, cudaDeviceSynchronize());  // the subspace copies are complete
  if (rc != ZGR_OK) {
    zgr_destroy(ctx);
    return rc;
  }
  ctx->sticky = 0;
  *out = ctx;
  return ZGR_OK;
}

int zgr_perturb(zgr_ctx* ctx, uint64_t seed, double scale, void* stream) {
  if (!ctx || !is_finite(scale)) return ZGR_EINVAL;
  if (ctx->sticky) return ctx->sticky;
  if (!on_ctx_device(ctx)) return ZGR_EINVAL;
  if (!ctx->ledger.empty() && !(ctx->ledger.size() == 1 && ctx->ledger.count(seed) == 1)) return ZGR_ESTATE;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  int rc = flush_descs(ctx, st);
  if (rc != ZGR_OK) return rc;
  // the first perturbation under a seed also keeps the norm bookkeeping when that is switched on
  const bool keep = ctx->stats_on && ctx->ledger.empty() && scale != 0.0 && sweep_stats_possible(ctx);
  if (keep) {
    rc = prepare_sweep_stats(ctx);
    if (rc != ZGR_OK) return rc;
    ctx->held_valid = false;
  }
  rc = sweep(ctx, ctx->groups, ctx->d_descs, 1, &seed, &scale, st, 0, -1, keep);
  if (rc != ZGR_OK) return rc;
  if (keep) {
    ctx->held_valid = true;
    ctx->held_seed = seed;
    ctx->held_c = scale;
  }
  ledger_add(ctx, seed, scale);
  return ZGR_OK;
}

int zgr_restore_update(zgr_ctx* ctx, uint64_t seed, double loss_plus, double loss_minus, double lr, void* stream) {
  if (!ctx || !is_finite(loss_plus) || !is_finite(loss_minus) || !is_finite(lr)) return ZGR_EINVAL;
  if (ctx->sticky) return ctx->sticky;
  if (!on_ctx_device(ctx)) return ZGR_EINVAL;
  const auto active = ctx->ledger.find(seed);
  if (active == ctx->ledger.end()) return ZGR_ESTATE;
  // Eq. (grad): projected gradient; Algorithm 1 "Update": W <- W - eta g z, fused with the restore
  const double g = (loss_plus - loss_minus) / (2.0 * ctx->cfg.eps);
  const double c = -active->second - lr * g;
  if (!is_finite(c)) return ZGR_EINVAL;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  int rc = flush_descs(ctx, st);
  if (rc != ZGR_OK) return rc;
  rc = sweep(ctx, ctx->groups, ctx->d_descs, 1, &seed, &c, st);
  if (rc != ZGR_OK) return rc;
  ctx->ledger.erase(seed);
  ctx->last_seed = seed;
  return ZGR_OK;
}

int zgr_sweep_multi(zgr_ctx* ctx, int32_t n, const uint64_t* seeds, const double* coeffs, void* stream) {
  if (!ctx || !seeds || !coeffs || n < 1 || n > ZGR_MAX_SEEDS) return ZGR_EINVAL;
  for (int32_t i = 0; i < n; ++i) {
    if (!is_finite(coeffs[i])) return ZGR_EINVAL;
    for (int32_t j = 0; j < i; ++j)
      if (seeds[j] == seeds[i]) return ZGR_EINVAL;
  }
  if (ctx->sticky) return ctx->sticky;
  if (!on_ctx_device(ctx)) return ZGR_EINVAL;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  int rc = flush_descs(ctx, st);
  if (rc != ZGR_OK) return rc;
  std::vector<Group>& groups = n > 1 ? multi_groups(ctx, n, &rc) : ctx->groups;
  if (rc != ZGR_OK) return rc;
  rc = sweep(ctx, groups, ctx->d_descs, n, seeds, coeffs, st);
  if (rc != ZGR_OK) return rc;
  for (int32_t i = 0; i < n; ++i) ledger_add(ctx, seeds[i], coeffs[i]);
  return ZGR_OK;
}

int zgr_restore_update_multi(zgr_ctx* ctx, int32_t n, const uint64_t* seeds, const double* loss_plus, const double* loss_minus, double lr,
                             void* stream) {
  if (!ctx || !seeds || !loss_plus || !loss_minus || n < 1 || n > ZGR_MAX_SEEDS || !is_finite(lr)) return ZGR_EINVAL;
  double c[ZGR_MAX_SEEDS];
  for (int32_t i = 0; i < n; ++i) {
    if (!is_finite(loss_plus[i]) || !is_finite(loss_minus[i])) return ZGR_EINVAL;
    for (int32_t j = 0; j < i; ++j)
      if (seeds[j] == seeds[i]) return ZGR_EINVAL;
    // Eq. (grad) per seed; Algorithm 1 "Recover gradient" sums g_t z_t over the seeds, "Update" applies it
    const double g = (loss_plus[i] - loss_minus[i]) / (2.0 * ctx->cfg.eps);
    const auto it = ctx->ledger.find(seeds[i]);
    c[i] = -(it == ctx->ledger.end() ? 0.0 : it->second) - lr * g;
    if (!is_finite(c[i])) return ZGR_EINVAL;
  }
  if (ctx->sticky) return ctx->sticky;
  if (!on_ctx_device(ctx)) return ZGR_EINVAL;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  int rc = flush_descs(ctx, st);
  if (rc != ZGR_OK) return rc;
  std::vector<Group>& groups = n > 1 ? multi_groups(ctx, n, &rc) : ctx->groups;
  if (rc != ZGR_OK) return rc;
  rc = sweep(ctx, groups, ctx->d_descs, n, seeds, c, st);
  if (rc != ZGR_OK) return rc;
  for (int32_t i = 0; i < n; ++i) ctx->ledger.erase(seeds[i]);
  ctx->last_seed = seeds[n - 1];
  return ZGR_OK;
}

int zgr_set_alpha(zgr_ctx* ctx, double alpha) {
  if (!ctx || !(alpha >= 0.0 && alpha <= 1.0)) return ZGR_EINVAL;
  if (ctx->sticky) return ctx->sticky;
  if (!ctx->ledger.empty()) return ZGR_ESTATE;
  // The kernels serving each tensor were chosen at zgr_init; a context built with alpha = 1 (no guided
  // part at all) has no tensor-core operands and keeps serving every tensor without its subspace.
  if (ctx->guided_at_init == false && alpha < 1.0 && ctx->K > 0) return ZGR_ESTATE;
  set_mixing(ctx, alpha);
  ctx->held_valid = false;
  return ZGR_OK;
}

int zgr_adapt_alpha(zgr_ctx* ctx, const double* stats, double alpha_min, double alpha_max, double eta, double* alpha_out) {
  if (!ctx || !stats || !alpha_out) return ZGR_EINVAL;
  if (!(alpha_min >= 0.0 && alpha_min <= alpha_max && alpha_max <= 1.0) || !(eta >= 0.0 && eta <= 1.0)) return ZGR_EINVAL;
  if (ctx->sticky) return ctx->sticky;
  if (!ctx->ledger.empty()) return ZGR_ESTATE;
  const double alpha_old = ctx->cfg.alpha;
  *alpha_out = alpha_old;
  // Energy of each part per unit of its mixing weight, from the norms measured under the current (a, b):
  // sum (a Z)^2 / a^2 per parameter and sum (b U G)^2 / b^2 per guided coefficient.  Eq. (perturbation) gives
  // the parts the weights alpha/d and (1 - alpha)/K (times d in the unit normalisation), so their energies
  // are equal where alpha / (1 - alpha) = e_g / e_iso.  A part that is switched off cannot be measured:
  // the ratio then stays as it is.
  if (ctx->a == 0.0 || ctx->b == 0.0 || ctx->K == 0) return ZGR_OK;
  double iso = 0.0, guided = 0.0;
  for (size_t l = 0; l < ctx->descs.size(); ++l) {
    if (!is_finite(stats[3 * l]) || !is_finite(stats[3 * l + 1]) || stats[3 * l] < 0.0 || stats[3 * l + 1] < 0.0) return ZGR_EINVAL;
    iso += stats[3 * l];
    guided += stats[3 * l + 1];
  }
  const double e_iso = iso / (ctx->a * ctx->a) / static_cast<double>(ctx->d);
  const double e_g = guided / (ctx->b * ctx->b) / static_cast<double>(ctx->K);
  if (!(e_iso + e_g > 0.0)) return ZGR_OK;
  double alpha = (1.0 - eta) * alpha_old + eta * (e_g / (e_iso + e_g));
  alpha = std::min(std::max(alpha, alpha_min), alpha_max);
  set_mixing(ctx, alpha);
  ctx->held_valid = false;
  *alpha_out = alpha;
  return ZGR_OK;
}

int zgr_set_coeffs_dtc_rows(zgr_ctx* ctx, int32_t tensor, const int8_t* q, const float* scale, const float* zero, int32_t bits, int32_t n_rows) {
  if (!ctx || tensor < 0 || tensor >= static_cast<int32_t>(ctx->descs.size())) return ZGR_EINVAL;
  if (!q || !scale || (bits != 8 && bits != 4)) return ZGR_EINVAL;
  TensorDesc& td = ctx->descs[static_cast<size_t>(tensor)];
  if (td.rank == 0 || n_rows < 1 || n_rows > td.rank) return ZGR_EINVAL;
  if (!ctx->ledger.empty()) return ZGR_ESTATE;
  td.q = q;
  td.qscale = scale;
  td.qzero = zero;
  td.qbits = bits;
  td.qrows = n_rows;
  ctx->descs_dirty = true;
  ctx->held_valid = false;
  return ZGR_OK;
}

int zgr_set_coeffs_dtc(zgr_ctx* ctx, int32_t tensor, const int8_t* q, const float* scale, const float* zero, int32_t bits) {
  if (!ctx || tensor < 0 || tensor >= static_cast<int32_t>(ctx->descs.size())) return ZGR_EINVAL;
  return zgr_set_coeffs_dtc_rows(ctx, tensor, q, scale, zero, bits, ctx->descs[static_cast<size_t>(tensor)].rank);
}

int zgr_perturb_layers(zgr_ctx* ctx, uint64_t seed, double scale, int32_t n_layers, const int32_t* layer_end, int32_t n_deliveries,
                       const zgr_coeff_delivery* deliveries, void* stream, void* copy_stream) {
  if (!ctx || !is_finite(scale) || n_layers < 1 || !layer_end || n_deliveries < 0 || (n_deliveries > 0 && !deliveries)) return ZGR_EINVAL;
  const int32_t n = static_cast<int32_t>(ctx->descs.size());
  for (int32_t L = 0; L < n_layers; ++L)
    if (layer_end[L] <= (L ? layer_end[L - 1] : 0) || layer_end[L] > n) return ZGR_EINVAL;
  if (layer_end[n_layers - 1] != n) return ZGR_EINVAL;
  // which layer each delivery belongs to; every delivery must name a tensor whose compressed coefficients are set
  std::vector<std::vector<int32_t>> by_layer(static_cast<size_t>(n_layers));
  std::vector<char> seen(static_cast<size_t>(n), 0);
  for (int32_t i = 0; i < n_deliveries; ++i) {
    const zgr_coeff_delivery& d = deliveries[i];
    if (d.tensor < 0 || d.tensor >= n || seen[static_cast<size_t>(d.tensor)] || (!d.q && !d.U)) return ZGR_EINVAL;
    seen[static_cast<size_t>(d.tensor)] = 1;
    const TensorDesc& td = ctx->descs[static_cast<size_t>(d.tensor)];
    if (d.q && (!d.scale || td.q == nullptr || (d.zero != nullptr) != (td.qzero != nullptr))) return ZGR_EINVAL;
    if (!d.q && (d.scale || d.zero)) return ZGR_EINVAL;
    if (d.U && td.rank == 0) return ZGR_EINVAL;
    const int32_t L = static_cast<int32_t>(std::upper_bound(layer_end, layer_end + n_layers, d.tensor) - layer_end);
    by_layer[static_cast<size_t>(L)].push_back(i);
  }
  if (ctx->sticky) return ctx->sticky;
  if (!on_ctx_device(ctx)) return ZGR_EINVAL;
  if (!ctx->ledger.empty() && (n_deliveries > 0 || !(ctx->ledger.size() == 1 && ctx->ledger.count(seed) == 1))) return ZGR_ESTATE;
  cudaStream_t st = static_cast<cudaStream_t>(stream), cs = static_cast<cudaStream_t>(copy_stream);
  int rc = flush_descs(ctx, st);
  if (rc != ZGR_OK) return rc;
  if (!ctx->aux_stream) {
    rc = check(ctx, cudaStreamCreateWithFlags(&ctx->aux_stream, cudaStreamNonBlocking));
    if (rc != ZGR_OK) return rc;
  }
  while (ctx->layer_events.size() < static_cast<size_t>(n_layers) + 2) {
    cudaEvent_t e = nullptr;
    rc = check(ctx, cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    if (rc != ZGR_OK) return rc;
    ctx->layer_events.push_back(e);
  }
  if (n_deliveries > 0) {
    // The copies may not overtake work already enqueued on `stream` that still reads the destination buffers.
    rc = check(ctx, cudaEventRecord(ctx->layer_events[static_cast<size_t>(n_layers)], st));
    if (rc == ZGR_OK) rc = check(ctx, cudaStreamWaitEvent(cs, ctx->layer_events[static_cast<size_t>(n_layers)], 0));
    if (rc != ZGR_OK) return rc;
    // All copies are enqueued up front, layer by layer: the copy engine runs ahead of the sweeps as far as it can,
    // so layer l + 1 (and later ones) travel while layer l is swept (Sec. 3.3).
    for (int32_t L = 0; L < n_layers; ++L) {
      if (by_layer[static_cast<size_t>(L)].empty()) continue;
      for (int32_t i : by_layer[static_cast<size_t>(L)]) {
        const zgr_coeff_delivery& d = deliveries[i];
        const TensorDesc& td = ctx->descs[static_cast<size_t>(d.tensor)];
        const size_t row_bytes = td.qbits == 4 ? static_cast<size_t>((td.cols + 1) / 2) : static_cast<size_t>(td.cols);
        if (d.q) {
          rc = check(ctx, cudaMemcpyAsync(const_cast<int8_t*>(td.q), d.q, row_bytes * static_cast<size_t>(td.qrows), cudaMemcpyHostToDevice, cs));
          if (rc == ZGR_OK)
            rc = check(ctx, cudaMemcpyAsync(const_cast<float*>(td.qscale), d.scale, sizeof(float) * static_cast<size_t>(td.qrows), cudaMemcpyHostToDevice, cs));
          if (rc == ZGR_OK && d.zero)
            rc = check(ctx, cudaMemcpyAsync(const_cast<float*>(td.qzero), d.zero, sizeof(float) * static_cast<size_t>(td.qrows), cudaMemcpyHostToDevice, cs));
        }
        if (rc == ZGR_OK && d.U)
          rc = check(ctx, cudaMemcpyAsync(const_cast<float*>(td.U), d.U, sizeof(float) * static_cast<size_t>(td.rows) * td.rank, cudaMemcpyHostToDevice, cs));
        if (rc != ZGR_OK) return rc;
      }
      rc = check(ctx, cudaEventRecord(ctx->layer_events[static_cast<size_t>(L)], cs));
      if (rc != ZGR_OK) return rc;
    }
  }
  const bool keep = ctx->stats_on && ctx->ledger.empty() && scale != 0.0 && sweep_stats_possible(ctx);
  if (keep) {
    rc = prepare_sweep_stats(ctx);
    if (rc != ZGR_OK) return rc;
  }
  ctx->held_valid = false;     // (a delivery changes the coefficients that earlier norms were taken with)
  // Layers touch disjoint tensors, so consecutive layers need no ordering between them: even layers run on the
  // caller's stream, odd ones on a stream of the library's, and the blocks of one layer's kernels start on the
  // SMs that the previous layer's last blocks have not reached any more.  The library's stream starts behind the
  // work already on the caller's stream, and the caller's stream ends by waiting for it.
  cudaEvent_t ev_begin = ctx->layer_events[static_cast<size_t>(n_layers) + 1];
  std::vector<int32_t> jobs;
  rc = check(ctx, cudaEventRecord(ev_begin, st));
  if (rc == ZGR_OK) rc = check(ctx, cudaStreamWaitEvent(ctx->aux_stream, ev_begin, 0));
  if (rc != ZGR_OK) return rc;
  for (int32_t L = 0; L < n_layers; ++L) {
    cudaStream_t ls = (L & 1) ? ctx->aux_stream : st;
    if (n_deliveries > 0 && !by_layer[static_cast<size_t>(L)].empty()) {
      rc = check(ctx, cudaStreamWaitEvent(ls, ctx->layer_events[static_cast<size_t>(L)], 0));
      if (rc != ZGR_OK) return rc;
      // the delivered subspaces, split for the tensor cores: one launch per run of neighbouring jobs (all of a layer, as a rule)
      jobs.clear();
      for (int32_t i : by_layer[static_cast<size_t>(L)]) {
        TensorDesc& td = ctx->descs[static_cast<size_t>(deliveries[i].tensor)];
        if (!deliveries[i].U) continue;
        if (td.Ufrag != nullptr && !td.umma) rc = make_fragments(ctx, td, ls);
        if (rc != ZGR_OK) return rc;
        if (ctx->split_job[static_cast<size_t>(deliveries[i].tensor)] >= 0) jobs.push_back(ctx->split_job[static_cast<size_t>(deliveries[i].tensor)]);
      }
      std::sort(jobs.begin(), jobs.end());
      for (size_t i = 0, end; i < jobs.size(); i = end) {
        for (end = i + 1; end < jobs.size() && jobs[end] == jobs[end - 1] + 1; ++end) {}
        rc = split_jobs(ctx, jobs[i], static_cast<int>(end - i), ls);
        if (rc != ZGR_OK) return rc;
      }
    }
    rc = sweep(ctx, ctx->groups, ctx->d_descs, 1, &seed, &scale, ls, L ? layer_end[L - 1] : 0, layer_end[L], keep);
    if (rc != ZGR_OK) return rc;   // (a failure here leaves the earlier layers swept: the context is sticky-failed by check())
  }
  if (n_layers > 1) {
    rc = check(ctx, cudaEventRecord(ev_begin, ctx->aux_stream));
    if (rc == ZGR_OK) rc = check(ctx, cudaStreamWaitEvent(st, ev_begin, 0));
    if (rc != ZGR_OK) return rc;
  }
  if (keep) {
    ctx->held_valid = true;
    ctx->held_seed = seed;
    ctx->held_c = scale;
  }
  ledger_add(ctx, seed, scale);
  return ZGR_OK;
}

int zgr_clear_coeffs(zgr_ctx* ctx, int32_t tensor) {
  if (!ctx || tensor < 0 || tensor >= static_cast<int32_t>(ctx->descs.size())) return ZGR_EINVAL;
  TensorDesc& td = ctx->descs[static_cast<size_t>(tensor)];
  if (td.rank == 0) return ZGR_EINVAL;
  if (!ctx->ledger.empty()) return ZGR_ESTATE;
  td.q = nullptr;
  td.qscale = nullptr;
  td.qzero = nullptr;
  td.qrows = 0;
  ctx->descs_dirty = true;
  ctx->held_valid = false;
  return ZGR_OK;
}

int zgr_get_stats(zgr_ctx* ctx, uint64_t seed, double* out, void* stream) {
  if (!ctx || !out) return ZGR_EINVAL;
  if (ctx->sticky) return ctx->sticky;
  if (!on_ctx_device(ctx)) return ZGR_EINVAL;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  int rc = flush_descs(ctx, st);
  if (rc != ZGR_OK) return rc;
  const size_t n = ctx->descs.size();
  if (ctx->held_valid && ctx->held_seed == seed) {
    // The first perturbation under this seed kept the bookkeeping: add up its partial sums (fixed order) and
    // read them back; they are the norms of c z, c being that perturbation's coefficient.
    rc = check(ctx, launch_stats_finish(ctx->d_ranges_sweep, static_cast<int>(n), ctx->d_stats, st));
    if (rc == ZGR_OK) ctx->launches++;
    if (rc == ZGR_OK) rc = check(ctx, cudaMemcpyAsync(out, ctx->d_stats, 3 * n * sizeof(double), cudaMemcpyDeviceToHost, st));
    if (rc == ZGR_OK) rc = check(ctx, cudaStreamSynchronize(st));
    if (rc != ZGR_OK) return rc;
    const double inv = 1.0 / (ctx->held_c * ctx->held_c);
    for (size_t i = 0; i < 3 * n; ++i) out[i] *= inv;
    return ZGR_OK;
  }
  // A pass of its own: regenerate Z and U G for `seed` without touching the weights.
  rc = prepare_sweep_stats(ctx);      // (the tcgen05 groups leave their partial sums in the slots of the sweep plan)
  if (rc != ZGR_OK) return rc;
  ctx->held_valid = false;
  if (!ctx->stats_planned) {
    // tensors served by the tcgen05 kernel reuse its work items; all others get a generic tiling (strips of 64 columns)
    int64_t total = ctx->d;
    int64_t target = std::min<int64_t>(std::max<int64_t>(total / (static_cast<int64_t>(ctx->sm_count) * 64), 4096), 131072);
    ctx->stats_first.assign(n + 1, 0);
    for (size_t l = 0; l < n; ++l) {
      const TensorDesc& t = ctx->descs[l];
      ctx->stats_first[l] = static_cast<int32_t>(ctx->stats_items.size());
      if (t.umma && ctx->guided_at_init) continue;
      for (int64_t c0 = 0; c0 < t.cols; c0 += 64) {
        const int ncols = static_cast<int>(std::min<int64_t>(64, t.cols - c0));
        const int64_t nrows = std::max<int64_t>(1, target / ncols);
        for (int64_t r0 = 0; r0 < t.rows; r0 += nrows)
          ctx->stats_items.push_back(WorkItem{static_cast<int32_t>(l), ncols, r0, std::min(nrows, t.rows - r0), c0});
      }
    }
    ctx->stats_first[n] = static_cast<int32_t>(ctx->stats_items.size());
    if (!ctx->stats_items.empty()) {
      rc = dev_alloc(ctx, &ctx->d_stats_items, ctx->stats_items.size());
      if (rc == ZGR_OK)
        rc = check(ctx, cudaMemcpy(ctx->d_stats_items, ctx->stats_items.data(), ctx->stats_items.size() * sizeof(WorkItem), cudaMemcpyHostToDevice));
      if (rc != ZGR_OK) return rc;
    }
    rc = alloc_slots(ctx, &ctx->d_stats_slots, ctx->stats_items.size());
    if (rc != ZGR_OK) return rc;
    std::vector<StatRange> ranges(n);
    for (size_t l = 0; l < n; ++l) {
      ranges[l] = StatRange{ctx->d_stats_slots, ctx->stats_first[l], ctx->stats_first[l + 1] - ctx->stats_first[l]};
      if (ctx->descs[l].umma && ctx->guided_at_init)
        for (const Group& g : ctx->groups)
          if (g.kc.path == PATH_UMMA && g.first_item[l + 1] > g.first_item[l])
            ranges[l] = StatRange{g.d_item_stats, g.first_item[l], g.first_item[l + 1] - g.first_item[l]};
    }
    rc = dev_alloc(ctx, &ctx->d_ranges_pass, n);
    if (rc == ZGR_OK) rc = check(ctx, cudaMemcpy(ctx->d_ranges_pass, ranges.data(), n * sizeof(StatRange), cudaMemcpyHostToDevice));
    if (rc != ZGR_OK) return rc;
    ctx->stats_planned = true;
  }
  SweepParams p;
  std::memset(&p, 0, sizeof(p));
  p.n_terms = 1;
  p.term[0].keys = make_keys(seed);
  p.term[0].iso = make_scale(ctx->a, ctx->cfg.bits_per_normal);
  p.unit = make_scale(1.0, ctx->cfg.bits_per_normal);
  p.tensors = ctx->d_descs;
  p.items = ctx->d_stats_items;
  p.n_items = static_cast<int32_t>(ctx->stats_items.size());
  p.term[0].cb = static_cast<float>(ctx->b);
  p.kshift = kshift_for(std::fabs(ctx->b));
  p.item_stats = ctx->d_stats_slots;
  p.item_base = 0;
  if (p.n_items > 0) {
    const int grid = static_cast<int>(std::min<int64_t>(p.n_items, static_cast<int64_t>(ctx->sm_count) * 4));
    rc = check(ctx, launch_stats(ctx->cfg.bits_per_normal, p, grid, st));
    if (rc != ZGR_OK) return rc;
    ctx->launches++;
  }
  for (const Group& g : ctx->groups) {
    if (g.kc.path != PATH_UMMA || g.items.empty()) continue;
    p.items = g.d_items;
    p.n_items = static_cast<int32_t>(g.items.size());
    p.item_stats = g.d_item_stats;
    rc = check(ctx, launch_stats_umma(g.kc, p, ctx->d_tmaps, ctx->d_err, g.grid, st));
    if (rc != ZGR_OK) return rc;
    ctx->launches++;
  }
  rc = check(ctx, launch_stats_finish(ctx->d_ranges_pass, static_cast<int>(n), ctx->d_stats, st));
  if (rc != ZGR_OK) return rc;
  ctx->launches++;
  rc = check(ctx, cudaMemcpyAsync(out, ctx->d_stats, 3 * n * sizeof(double), cudaMemcpyDeviceToHost, st));
  if (rc != ZGR_OK) return rc;
  return check(ctx, cudaStreamSynchronize(st));
}

int zgr_enable_stats(zgr_ctx* ctx, int32_t enable) {
  if (!ctx) return ZGR_EINVAL;
  ctx->stats_on = enable != 0;     // norms already held stay available until something they depend on changes
  // the slots of the partial sums, here rather than inside the first perturbation
  if (ctx->stats_on && ctx->sticky == 0 && on_ctx_device(ctx) && sweep_stats_possible(ctx)) return prepare_sweep_stats(ctx);
  return ZGR_OK;
}

int zgr_debug_philox(zgr_ctx* ctx, uint64_t seed, int32_t tensor, int32_t tag, uint64_t first_block, int64_t n_blocks, uint32_t* dev_out,
                     void* stream) {
  if (!ctx || !dev_out || n_blocks < 0 || tensor < 0 || tag < 0) return ZGR_EINVAL;
  if (reinterpret_cast<uintptr_t>(dev_out) % 16 != 0) return ZGR_EINVAL;
  if (ctx->sticky) return ctx->sticky;
  if (!on_ctx_device(ctx)) return ZGR_EINVAL;
  if (n_blocks == 0) return ZGR_OK;
  const int rc = check(ctx, launch_philox_blocks(make_keys(seed), static_cast<uint32_t>(tensor), static_cast<uint32_t>(tag), first_block, n_blocks,
                                                 dev_out, static_cast<cudaStream_t>(stream)));
  if (rc == ZGR_OK) ctx->launches++;
  return rc;
}

int zgr_debug_z(zgr_ctx* ctx, uint64_t seed, int32_t tensor, float* dev_out, void* stream) {
  if (!ctx || !dev_out || tensor < 0 || tensor >= static_cast<int32_t>(ctx->descs.size())) return ZGR_EINVAL;
  if (reinterpret_cast<uintptr_t>(dev_out) % 4 != 0) return ZGR_EINVAL;
  if (ctx->sticky) return ctx->sticky;
  if (!on_ctx_device(ctx)) return ZGR_EINVAL;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (ctx->descs[static_cast<size_t>(tensor)].umma) {
    const int rcf = make_fragments(ctx, ctx->descs[static_cast<size_t>(tensor)], st);
    if (rcf != ZGR_OK) return rcf;
  }
  // a one-tensor model whose weights are the zeroed output buffer, swept once with scale 1
  std::vector<TensorDesc> one(1, ctx->descs[static_cast<size_t>(tensor)]);
  one[0].data = dev_out;
  if (one[0].dtype != ZGR_F32) one[0].tile = one[0].staged = 0;      // (its kernels read 16-bit weights)
  const size_t owned_before = ctx->owned.size();
  int rc = ZGR_OK;
  if (one[0].staged) {
    // the tensor's own kernel on the image: its maps of U, and new ones of the weights
    const size_t n_maps = static_cast<size_t>(n_weight_maps(one[0]));
    std::vector<CUtensorMap> maps(n_maps);
    CUtensorMap* d_maps = nullptr;
    if ((reinterpret_cast<uintptr_t>(dev_out) & 15) != 0 || !make_weight_maps(maps.data(), one[0], dev_out, 4)) {
      one[0].tile = one[0].staged = 0;                 // (an image that TMA cannot address: one element per thread)
    } else {
      rc = dev_alloc(ctx, &d_maps, n_maps + 3);
      if (rc == ZGR_OK) rc = check(ctx, cudaMemcpy(d_maps, maps.data(), n_maps * sizeof(CUtensorMap), cudaMemcpyHostToDevice));
      if (rc == ZGR_OK) rc = check(ctx, cudaMemcpy(d_maps + n_maps, static_cast<const CUtensorMap*>(one[0].maps) + n_maps, 3 * sizeof(CUtensorMap), cudaMemcpyDeviceToDevice));
      one[0].maps = d_maps;
    }
  }
  std::vector<Group> groups;
  const bool guided_on = ctx->guided_at_init;
  plan(one, std::vector<int>(1, 0), guided_on, ctx->cfg.bits_per_normal, ctx->sm_count, groups, ZGR_F32);
  TensorDesc* d_one = nullptr;
  if (rc == ZGR_OK) rc = dev_alloc(ctx, &d_one, 1);
  if (rc == ZGR_OK) rc = check(ctx, cudaMemcpy(d_one, one.data(), sizeof(TensorDesc), cudaMemcpyHostToDevice));
  if (rc == ZGR_OK) rc = upload_groups(ctx, groups);
  if (rc == ZGR_OK) rc = check(ctx, cudaMemsetAsync(dev_out, 0, static_cast<size_t>(one[0].rows * one[0].cols) * sizeof(float), st));
  const double one_scale = 1.0;
  if (rc == ZGR_OK) rc = sweep(ctx, groups, d_one, 1, &seed, &one_scale, st, 0, -1, false, ctx->d_tmaps + 3 * tensor);
  if (rc == ZGR_OK) rc = check(ctx, cudaStreamSynchronize(st));
  for (size_t i = owned_before; i < ctx->owned.size(); ++i) cudaFree(ctx->owned[i]);
  ctx->owned.resize(owned_before);
  return rc;
}

int zgr_debug_z_tcgen05(zgr_ctx* ctx, uint64_t seed, int32_t tensor, float* dev_out, void* stream) {
  if (!ctx || !dev_out || tensor < 0 || tensor >= static_cast<int32_t>(ctx->descs.size())) return ZGR_EINVAL;
  if (reinterpret_cast<uintptr_t>(dev_out) % 16 != 0) return ZGR_EINVAL;
  if (ctx->sticky) return ctx->sticky;
  if (!on_ctx_device(ctx)) return ZGR_EINVAL;
  const TensorDesc& cur = ctx->descs[static_cast<size_t>(tensor)];
  if (!cur.umma || !ctx->guided_at_init) return ZGR_ESTATE;   // the sweeps do not serve this tensor with the tcgen05 kernel
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  int rc = flush_descs(ctx, st);
  if (rc != ZGR_OK) return rc;
  // A one-tensor model whose weights are a zeroed 16-bit image, swept once with coefficient 1 by the tcgen05
  // kernel itself; its fp32 results go to dev_out instead of being rounded into the image.
  const size_t owned_before = ctx->owned.size();
  const size_t numel = static_cast<size_t>(cur.rows * cur.cols);
  uint16_t* image = nullptr;
  CUtensorMap* d_maps = nullptr;
  TensorDesc* d_one = nullptr;
  std::vector<Group> groups;
  rc = dev_alloc(ctx, &image, numel);
  if (rc == ZGR_OK) rc = check(ctx, cudaMemsetAsync(image, 0, numel * sizeof(uint16_t), st));
  CUtensorMap maps[3];
  if (rc == ZGR_OK) {
    maps[1] = ctx->tmaps[static_cast<size_t>(3 * tensor + 1)];
    maps[2] = ctx->tmaps[static_cast<size_t>(3 * tensor + 2)];
    if (!make_map_16bit(&maps[0], image, cur.rows, cur.cols, 64)) rc = check(ctx, cudaErrorUnknown);
  }
  if (rc == ZGR_OK) rc = dev_alloc(ctx, &d_maps, 3);
  if (rc == ZGR_OK) rc = check(ctx, cudaMemcpyAsync(d_maps, maps, sizeof(maps), cudaMemcpyHostToDevice, st));
  std::vector<TensorDesc> one(1, cur);
  one[0].data = image;
  if (rc == ZGR_OK) rc = dev_alloc(ctx, &d_one, 1);
  if (rc == ZGR_OK) rc = check(ctx, cudaMemcpyAsync(d_one, one.data(), sizeof(TensorDesc), cudaMemcpyHostToDevice, st));
  if (rc == ZGR_OK) {
    plan(one, std::vector<int>(1, 0), true, ctx->cfg.bits_per_normal, ctx->sm_count, groups);
    rc = upload_groups(ctx, groups);
  }
  if (rc == ZGR_OK) {
    SweepParams p;
    std::memset(&p, 0, sizeof(p));
    p.term[0].keys = make_keys(seed);
    p.term[0].iso = make_scale(ctx->a, ctx->cfg.bits_per_normal);
    p.term[0].cb = static_cast<float>(ctx->b);
    p.n_terms = 1;
    p.unit = make_scale(1.0, ctx->cfg.bits_per_normal);
    p.tensors = d_one;
    p.zout = dev_out;
    p.kshift = kshift_for(std::fabs(ctx->b));
    for (Group& g : groups) {
      if (g.items.empty()) continue;
      if (g.kc.path != PATH_UMMA) { rc = ZGR_ESTATE; break; }
      p.items = g.d_items;
      p.n_items = static_cast<int32_t>(g.items.size());
      rc = check(ctx, launch_debug_z_umma(g.kc, p, d_maps, ctx->d_err, g.grid, st));
      if (rc != ZGR_OK) break;
      ctx->launches++;
    }
  }
  const int rc_sync = check(ctx, cudaStreamSynchronize(st));
  if (rc == ZGR_OK) rc = rc_sync;
  for (size_t i = owned_before; i < ctx->owned.size(); ++i) cudaFree(ctx->owned[i]);
  ctx->owned.resize(owned_before);
  return rc;
}

int zgr_update_subspace(zgr_ctx* ctx, int32_t tensor, const float* U_src, int32_t src_is_host, void* stream) {
  if (!ctx || tensor < 0 || tensor >= static_cast<int32_t>(ctx->descs.size())) return ZGR_EINVAL;
  TensorDesc& td = ctx->descs[static_cast<size_t>(tensor)];
  if (td.rank == 0) return ZGR_EINVAL;
  if (ctx->sticky) return ctx->sticky;
  if (!on_ctx_device(ctx)) return ZGR_EINVAL;
  if (!ctx->ledger.empty()) return ZGR_ESTATE;
  ctx->held_valid = false;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  int rc = ZGR_OK;
  if (U_src != nullptr && U_src != td.U) {
    const size_t bytes = static_cast<size_t>(td.rows) * td.rank * sizeof(float);
    rc = check(ctx, cudaMemcpyAsync(const_cast<float*>(td.U), U_src, bytes, src_is_host ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice, st));
    if (rc != ZGR_OK) return rc;
  }
  return refresh_operands(ctx, tensor, st);
}

int zgr_build_subspace(zgr_ctx* ctx, int32_t tensor, const float* grads, int32_t src_is_host, void* stream) {
  if (!ctx || tensor < 0 || tensor >= static_cast<int32_t>(ctx->descs.size())) return ZGR_EINVAL;
  TensorDesc& td = ctx->descs[static_cast<size_t>(tensor)];
  if (td.rank == 0 || td.rows < td.rank) return ZGR_EINVAL;
  if (grads && reinterpret_cast<uintptr_t>(grads) % 4 != 0) return ZGR_EINVAL;
  if (ctx->sticky) return ctx->sticky;
  if (!on_ctx_device(ctx)) return ZGR_EINVAL;
  if (!ctx->ledger.empty()) return ZGR_ESTATE;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const size_t need = subspace_scratch_bytes(td.rows, td.rank, ctx->sm_count);
  if (need > ctx->qr_bytes) {
    void* q = nullptr;
    int rc = check(ctx, cudaMalloc(&q, need));
    if (rc != ZGR_OK) return rc;
    ctx->owned.push_back(q);          // an outgrown scratch buffer stays owned until zgr_destroy; work enqueued on it may still run
    rc = check(ctx, cudaMemsetAsync(q, 0, 512, st));
    if (rc != ZGR_OK) return rc;
    ctx->d_qr = q;
    ctx->qr_bytes = need;
  }
  if (!ctx->h_status) {
    const int rc = check(ctx, status_words().take(&ctx->h_status, &ctx->h_status_own));
    if (rc != ZGR_OK) return rc;
  }
  float* U = const_cast<float*>(td.U);
  const float* A = U;                  // NULL source: the gradient directions were written into the subspace buffer itself
  if (grads != nullptr && grads != td.U) {
    if (src_is_host) {
      const size_t bytes = static_cast<size_t>(td.rows) * td.rank * sizeof(float);
      const int rc = check(ctx, cudaMemcpyAsync(U, grads, bytes, cudaMemcpyHostToDevice, st));
      if (rc != ZGR_OK) return rc;
    } else {
      A = grads;
    }
  }
  ctx->held_valid = false;
  int rc;
  if (subspace_fused(td.rows, td.rank, ctx->sm_count)) {
    const int32_t job = ctx->split_job[static_cast<size_t>(tensor)];
    constexpr int kPending = INT32_MIN;
    volatile int* const h_status = ctx->h_status;
    *h_status = kPending;
    rc = check(ctx, launch_basis_fused(A, td.rows, td.rank, U, job >= 0 ? &ctx->split_jobs[static_cast<size_t>(job)] : nullptr, ctx->d_qr, ctx->h_status,
                                       ctx->sm_count, st));
    // The kernel writes the word when everything it does is visible, some microseconds before the driver would report the
    // stream idle; if it has not come after a while (a long queue, or a failed launch) the driver is asked.
    for (int spin = 0; rc == ZGR_OK && *h_status == kPending && spin < 1000000; ++spin) {}
    if (rc == ZGR_OK && *h_status == kPending) rc = check(ctx, cudaStreamSynchronize(st));
    if (rc != ZGR_OK) return rc;
    ctx->launches++;
    const int status = *h_status;
    if (status < 0) return check(ctx, cudaErrorLaunchTimeout);   // a barrier gave up: the basis may be partly written
    if (status > 0) return ZGR_EINVAL;                            // linearly dependent directions: nothing was written
    if (td.Ufrag == nullptr || td.umma) return ZGR_OK;
    rc = make_fragments(ctx, td, st);
    return rc == ZGR_OK ? check(ctx, cudaStreamSynchronize(st)) : rc;
  }
  int* d_status = nullptr;
  rc = check(ctx, launch_build_subspace(A, td.rows, td.rank, U, ctx->d_qr, &d_status, nullptr, st));
  if (rc != ZGR_OK) return rc;
  ctx->launches += 6;
  int status = 0;
  rc = check(ctx, cudaMemcpyAsync(&status, d_status, sizeof(int), cudaMemcpyDeviceToHost, st));
  if (rc == ZGR_OK) rc = check(ctx, cudaStreamSynchronize(st));
  if (rc != ZGR_OK) return rc;
  if (status != 0) return ZGR_EINVAL;  // linearly dependent directions: nothing was written
  // the new basis is in place: refresh the tensor-core operand copies exactly as for a delivered subspace (only now that the
  // status is known: a refused input leaves them alone too), and wait for them, which sweeps on any stream may read next
  rc = refresh_operands(ctx, tensor, st);
  return rc == ZGR_OK ? check(ctx, cudaStreamSynchronize(st)) : rc;
}

int zgr_debug_plan(const zgr_tensor* tensors, int32_t n, const zgr_config* cfg, int32_t sm_count, int32_t tcgen05, int32_t multi,
                   zgr_plan_item* out, int64_t max_items, int64_t* n_items) {
  if (!n_items || sm_count < 1 || max_items < 0 || (max_items > 0 && !out)) return ZGR_EINVAL;
  std::vector<TensorDesc> descs;
  std::vector<Group> groups;
  const int rc = plan_on_host(tensors, n, cfg, sm_count, tcgen05 != 0, multi != 0, descs, groups);
  if (rc != ZGR_OK) return rc;
  int64_t count = 0;
  for (const Group& g : groups)
    for (const WorkItem& w : g.items) {
      const auto [first, rows] = g.kc.path == PATH_ISO ? std::make_pair(w.row0_or_e0, w.nrows_or_count) : item_rows(descs[w.tensor], g.kc, w);
      if (count < max_items) out[count] = zgr_plan_item{g.kc.path, g.kc.kpad, w.tensor, w.ncols, first, rows, w.col0};
      ++count;
    }
  *n_items = count;
  return ZGR_OK;
}

int zgr_debug_plan_kernels(const zgr_tensor* tensors, int32_t n, const zgr_config* cfg, int32_t sm_count, int32_t tcgen05, int32_t multi, int32_t* kernels) {
  if (!kernels || sm_count < 1) return ZGR_EINVAL;
  std::vector<TensorDesc> descs;
  std::vector<Group> groups;
  const int rc = plan_on_host(tensors, n, cfg, sm_count, tcgen05 != 0, multi != 0, descs, groups);
  if (rc != ZGR_OK) return rc;
  for (const Group& g : groups)
    for (const WorkItem& w : g.items) kernels[w.tensor] = kernel_number(g.kc);
  return ZGR_OK;
}

int zgr_update_subspaces(zgr_ctx* ctx, int32_t n, const int32_t* tensors, const float* const* U_src, int32_t src_is_host, void* stream) {
  if (!ctx || !tensors || n < 1) return ZGR_EINVAL;
  std::vector<char> seen(ctx->descs.size(), 0);
  int n_jobs = 0;
  for (int32_t i = 0; i < n; ++i) {
    const int32_t l = tensors[i];
    if (l < 0 || l >= static_cast<int32_t>(ctx->descs.size()) || seen[static_cast<size_t>(l)]) return ZGR_EINVAL;
    seen[static_cast<size_t>(l)] = 1;
    if (ctx->descs[static_cast<size_t>(l)].rank == 0) return ZGR_EINVAL;
    n_jobs += ctx->split_job[static_cast<size_t>(l)] >= 0 ? 1 : 0;
  }
  if (ctx->sticky) return ctx->sticky;
  if (!on_ctx_device(ctx)) return ZGR_EINVAL;
  if (!ctx->ledger.empty()) return ZGR_ESTATE;
  ctx->held_valid = false;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // every tensor of the tcgen05 paths is listed: their operand copies are rebuilt by one launch after the copies
  const bool fused = n_jobs > 0 && n_jobs == ctx->n_split_jobs;
  for (int32_t i = 0; i < n; ++i) {
    const int32_t l = tensors[i];
    TensorDesc& td = ctx->descs[static_cast<size_t>(l)];
    const float* src = U_src ? U_src[i] : nullptr;
    if (src != nullptr && src != td.U) {
      const size_t bytes = static_cast<size_t>(td.rows) * td.rank * sizeof(float);
      const int rc = check(ctx, cudaMemcpyAsync(const_cast<float*>(td.U), src, bytes, src_is_host ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice, st));
      if (rc != ZGR_OK) return rc;
    }
    if (td.Ufrag != nullptr && !td.umma) {
      const int rc = make_fragments(ctx, td, st);
      if (rc != ZGR_OK) return rc;
    }
    const int32_t job = ctx->split_job[static_cast<size_t>(l)];
    if (job >= 0 && !fused) {
      const int rc = split_jobs(ctx, job, 1, st);
      if (rc != ZGR_OK) return rc;
    }
  }
  if (fused) {
    const int rc = split_jobs(ctx, 0, ctx->n_split_jobs, st);
    if (rc != ZGR_OK) return rc;
  }
  return ZGR_OK;
}

int zgr_profile(zgr_ctx* ctx, int32_t enable) {
  if (!ctx) return ZGR_EINVAL;
  ctx->profiling = enable != 0;
  return ZGR_OK;
}

int zgr_profile_read(zgr_ctx* ctx, zgr_kernel_time* out, int32_t max_entries, int32_t* n_entries) {
  if (!ctx || !out || !n_entries || max_entries < 0) return ZGR_EINVAL;
  if (ctx->sticky) return ctx->sticky;
  const int rc = check(ctx, cudaDeviceSynchronize());
  if (rc != ZGR_OK) return rc;
  int32_t n = 0;
  ctx->profiled.clear();
  for (std::vector<Group>* gs : {&ctx->groups, &ctx->groups_multi})
  for (Group& g : *gs) {
    if (g.timed.empty()) continue;
    double total = 0.0;
    for (auto& ev : g.timed) {
      float ms = 0.0f;
      if (cudaEventElapsedTime(&ms, ev.first, ev.second) == cudaSuccess) total += ms;
      cudaEventDestroy(ev.first);
      cudaEventDestroy(ev.second);
    }
    if (n < max_entries) {
      zgr_kernel_time& o = out[n];
      o.path = g.kc.path;
      o.dtype = g.kc.dtype;
      o.kpad = g.kc.kpad;
      o.launches = static_cast<int32_t>(g.timed.size());
      o.elements = g.elements;
      o.ms_total = total;
      ctx->profiled.push_back(kernel_number(g.kc));
      ++n;
    }
    g.timed.clear();
  }
  *n_entries = n;
  return ZGR_OK;
}

int zgr_profile_kernels(zgr_ctx* ctx, int32_t* kernels, int32_t max_entries, int32_t* n_entries) {
  if (!ctx || !kernels || !n_entries || max_entries < 0) return ZGR_EINVAL;
  *n_entries = std::min(max_entries, static_cast<int32_t>(ctx->profiled.size()));
  std::copy_n(ctx->profiled.begin(), *n_entries, kernels);
  return ZGR_OK;
}

int zgr_device_status(zgr_ctx* ctx, int32_t* code) {
  if (!ctx || !code) return ZGR_EINVAL;
  if (ctx->sticky) return ctx->sticky;
  int rc = check(ctx, cudaDeviceSynchronize());
  if (rc != ZGR_OK) return rc;
  int v = 0;
  rc = check(ctx, cudaMemcpy(&v, ctx->d_err, sizeof(int), cudaMemcpyDeviceToHost));
  if (rc != ZGR_OK) return rc;
  *code = v;
  if (v != 0) ctx->sticky = ZGR_ECUDA;   // a kernel gave up on a wait: its sweep is incomplete, the weights are not trustworthy
  return ZGR_OK;
}

int zgr_get_scalars(const zgr_ctx* ctx, double* a, double* b) {
  if (!ctx || !a || !b) return ZGR_EINVAL;
  *a = ctx->a;
  *b = ctx->b;
  return ZGR_OK;
}

int zgr_get_state(const zgr_ctx* ctx, int32_t* active, uint64_t* seed, double* net_scale) {
  if (!ctx || !active || !seed || !net_scale) return ZGR_EINVAL;
  *active = static_cast<int32_t>(ctx->ledger.size());
  const auto it = ctx->ledger.find(ctx->last_seed);
  *seed = ctx->last_seed;
  *net_scale = it == ctx->ledger.end() ? 0.0 : it->second;
  return ZGR_OK;
}

int zgr_debug_check_device(int32_t ctx_device, int32_t current_device) {
  return (ctx_device >= 0 && ctx_device == current_device) ? ZGR_OK : ZGR_EINVAL;
}

int64_t zgr_launch_count(const zgr_ctx* ctx) { return ctx ? ctx->launches : -1; }

void zgr_destroy(zgr_ctx* ctx) {
  if (!ctx) return;
  for (std::vector<Group>* gs : {&ctx->groups, &ctx->groups_multi})
    for (Group& g : *gs)
      for (auto& ev : g.timed) {
        cudaEventDestroy(ev.first);
        cudaEventDestroy(ev.second);
      }
  for (cudaEvent_t e : ctx->layer_events) cudaEventDestroy(e);
  if (ctx->aux_stream) cudaStreamDestroy(ctx->aux_stream);
  for (void* p : ctx->owned) cudaFree(p);
  status_words().give_back(ctx->h_status, ctx->h_status_own);
  delete ctx;
}

const char* zgr_strerror(int code) {
  switch (code) {
    case ZGR_OK: return "ok";
    case ZGR_EINVAL: return "invalid argument";
    case ZGR_ESTATE: return "call out of sequence (perturb / restore_update seeds do not match)";
    case ZGR_ECUDA: return "CUDA runtime error (no device, launch failure); the context is unusable";
    case ZGR_ENOMEM: return "out of device or host memory";
    case ZGR_ETOOBIG: return "tensor larger than the fixed scratch of the allocation-free entry point (ZGR_NOALLOC_MAX_TILES tiles of 1024 x 64)";
    default: return "unknown error code";
  }
}

}  // extern "C"
