// Host side of the tcgen05 GEMM: tensor-map encoding, tile selection, launch, and the
// stand-alone lp_gemm_bf16 entry point.
#include "gemm2q.cuh"
#include "gemmc.cuh"
#include "conv_wide.cuh"

#include <algorithm>
#include <atomic>
#include <cstdlib>
#include <mutex>

#include "common.h"

namespace lp {

// ---------------------------------------------------------------------------
// cuTensorMapEncodeTiled is a driver API; fetch it through the runtime so the library has
// no link-time dependency on libcuda.
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn get_encode_fn(std::string* err) {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  static std::string first_err;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    cudaError_t e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q);
    if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || p == nullptr) {
      first_err = std::string("cuTensorMapEncodeTiled unavailable: ") + cudaGetErrorString(e);
    } else {
      fn = reinterpret_cast<EncodeTiledFn>(p);
    }
  });
  if (!fn && err) *err = first_err;
  return fn;
}

int make_tmap_bf16_2d(CUtensorMap* out, const void* base, uint64_t inner, uint64_t outer, uint64_t pitch_elems,
                      uint32_t box_inner, uint32_t box_outer, std::string* err) {
  EncodeTiledFn fn = get_encode_fn(err);
  if (!fn) return LP_ERR_CUDA;
  if ((reinterpret_cast<uintptr_t>(base) & 15) || (pitch_elems & 7) || box_inner != 64 || box_outer > 256) {
    if (err) *err = "tensor map: base must be 16-byte aligned, pitch a multiple of 8 elements, box <= 256";
    return LP_ERR_INVALID_ARG;
  }
  cuuint64_t dims[2] = {inner, outer};
  cuuint64_t strides[1] = {pitch_elems * 2};
  cuuint32_t box[2] = {box_inner, box_outer};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    if (err) *err = "cuTensorMapEncodeTiled failed with CUresult " + std::to_string(int(r));
    return LP_ERR_CUDA;
  }
  return LP_OK;
}

// Row-major 2-D tensor of 4-byte (fp32) or 2-byte (bf16) elements moved in boxes of 32 columns:
// 128-byte rows with the 128-byte swizzle, or 64-byte rows with the 64-byte swizzle.
int make_tmap_rows32(CUtensorMap* out, const void* base, int elem_bytes, uint64_t inner, uint64_t outer,
                     uint64_t pitch_elems, uint32_t box_outer, std::string* err) {
  EncodeTiledFn fn = get_encode_fn(err);
  if (!fn) return LP_ERR_CUDA;
  if ((reinterpret_cast<uintptr_t>(base) & 15) || ((pitch_elems * elem_bytes) & 15) || box_outer > 256 ||
      (elem_bytes != 4 && elem_bytes != 2)) {
    if (err) *err = "tensor map: base and pitch must be 16-byte aligned, box <= 256";
    return LP_ERR_INVALID_ARG;
  }
  cuuint64_t dims[2] = {inner, outer};
  cuuint64_t strides[1] = {pitch_elems * elem_bytes};
  cuuint32_t box[2] = {32, box_outer};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(out, elem_bytes == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
                  const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  elem_bytes == 4 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    if (err) *err = "cuTensorMapEncodeTiled (update tile) failed with CUresult " + std::to_string(int(r));
    return LP_ERR_CUDA;
  }
  return LP_OK;
}

// NHWC bf16 tensor [N][H][W][C] with channel pitch `pitch_c` (multiple of 8): dimensions
// (C, W, H, N), box (64 channels, bw, bh, bn pixels).  Coordinates outside the tensor read zero.
int make_tmap_bf16_nhwc(CUtensorMap* out, const void* base, uint64_t C, uint64_t W, uint64_t H, uint64_t N,
                        uint64_t pitch_c, uint32_t bw, uint32_t bh, uint32_t bn, std::string* err, uint32_t step) {
  EncodeTiledFn fn = get_encode_fn(err);
  if (!fn) return LP_ERR_CUDA;
  if ((reinterpret_cast<uintptr_t>(base) & 15) || (pitch_c & 7) || step < 1 || bw * step > 256 || bh * step > 256 || bn > 256) {
    if (err) *err = "tensor map: base must be 16-byte aligned, channel pitch a multiple of 8, box <= 256";
    return LP_ERR_INVALID_ARG;
  }
  // step > 1: the box takes every step-th pixel in w and h (a strided convolution's input seen from a
  // box of its output pixels): the traversed extent is bw * step, of which ceil(. / step) = bw are loaded
  cuuint64_t dims[4] = {C, W, H, N};
  cuuint64_t strides[3] = {pitch_c * 2, W * pitch_c * 2, H * W * pitch_c * 2};
  cuuint32_t box[4] = {64, bw * step, bh * step, bn};
  cuuint32_t estr[4] = {1, step, step, 1};
  CUresult r = fn(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    if (err) *err = "cuTensorMapEncodeTiled (4-D) failed with CUresult " + std::to_string(int(r));
    return LP_ERR_CUDA;
  }
  return LP_OK;
}

// ---------------------------------------------------------------------------
static int g_force_bn = 0;
static int g_force_stages = 0;
static int g_force_splits = 0;
static int g_l2_ahead = 16;   // measured 0 / 8 / 16 / 32 / 64 k-blocks ahead: 47.0 / 46.2 / 45.2 / 47.0 / 50.8 us (256 x 4096 x 4096)
static int g_force_persistent = -1;   // -1 automatic, 0 one tile per CTA, 1 persistent CTAs
void gemm_set_tuning(int bn, int stages, int splits) {
  g_force_bn = bn;
  g_force_stages = stages;
  g_force_splits = splits >= 0 ? (splits & 0xFF) : 0;
  // bits 8-9 of the third tuning knob force the tile loop: 1 = one tile per CTA, 2 = persistent
  g_force_persistent = splits >= 0 ? ((splits >> 8) & 3) - 1 : -1;
  if (g_force_persistent > 1) g_force_persistent = -1;
}

// What lp_debug_last_contraction tells: the kernel form of this thread's latest contraction launch, its tile width, and
// the cluster size or pipeline depth where that is part of the choice.
struct LastContraction {
  const char* kernel;
  int tile, detail;
};
static thread_local LastContraction t_last = {"", 0, 0};
static void note_form(const char* kernel, int tile, int detail = 0) { t_last = {kernel, tile, detail}; }
const char* gemm_last_contraction() {
  static thread_local char text[96];
  if (t_last.detail > 0) snprintf(text, sizeof text, "%s %d x%d", t_last.kernel, t_last.tile, t_last.detail);
  else                   snprintf(text, sizeof text, "%s %d", t_last.kernel, t_last.tile);
  return t_last.tile == 0 ? "" : text;
}

static int sm_count() {
  static int n = 0;
  if (n == 0) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1)
      n = kSMs;
  }
  return n;
}

// Split-K factor.  Measured on B200 (M = 256, N = K = 4096): the split main loop is shorter
// but writing and re-reading the fp32 partial tiles costs more than it saves (25 us unsplit,
// 28 / 35 / 52 us at 2 / 4 / 8 splits), and under the stage scheduler other kernels fill the
// idle SMs anyway.  So the automatic choice is "off" for such shapes; the path is covered by the
// tests through lp_set_tuning.
int gemm_pick_splits(int M, int N, int K, int bn) {
  const int num_kb = (K + GEMM_BK - 1) / GEMM_BK;
  // The exception: a handful of tiles with a very long contraction (64 x 4096 x 25088: 32 tiles of
  // 392 k-blocks, one CTA streaming 6.4 MB of weights each): 145 us unsplit, 95 / 74 / 89 us at
  // 2 / 4 / 8 splits.
  const long long tiles = (long long)((M + GEMM_BM - 1) / GEMM_BM) * ((N + bn - 1) / bn);
  // Fewer tiles with longer contractions take more splits: about one CTA per SM, never fewer than 16 k-blocks per
  // split (a single 10-column tile over 100352 inputs, the classifier behind an unpooled 28 x 28 x 128 image: 24 splits
  // added by the last CTA of the tile 37 us, 98 added by a launch on all SMs 15; 64 x 300 x 24576 40 -> 15; at
  // least 32 k-blocks a split, or two CTAs per SM, are no better).
  const int automatic = (tiles <= 48 && num_kb >= 256) ? int(std::max<long long>(1, std::min<long long>(kSMs / tiles, num_kb / 16))) : 1;
  int s = g_force_splits > 0 ? g_force_splits : automatic;
  s = std::max(1, std::min(s, num_kb));
  const int per = (num_kb + s - 1) / s;
  return (num_kb + per - 1) / per;      // no empty split
}

// Outputs of few tiles: one tile per cluster, the contraction divided over its CTAs (gemmc.cuh).  Sets the tile width and
// returns the cluster size (1: undivided, in that kernel's form), or 0 where another form is the better one.  Rule, each side
// measured on calls that follow one another in a stream (us):
// * 64-column tiles while they fit one CTA on every SM (100 x 777 x 1003 6.1 against 7.3 with 128 columns, 700^3 6.9 / 7.9,
//   512 x 2048 x 2048 12.7 / 13.3; beyond that 128: 512 x 4096 x 4096 24.5 / 25.7);
// * up to four k-blocks of such a tile undivided: a barrier and a pass through distributed shared memory cost what
//   they save (128 x 256 x 256 one CTA a tile 4.6, two 4.9, four 4.8; 128 x 256 x 128 4.1, two 4.6) -- but not in a layer, whose
//   epilogue gains by the division (16 steps of the ragged GELU MLP 620, undivided 640);
// * else eight CTAs to a tile for a handful of tiles (128 x 64 x 1500 5.6, in quarters 6.2; 128 x 800 x 3000 on 13 tiles 7.5 / 8.3, but
//   x 784 6.1 / 5.7), four, or two, while that is at most one CTA per SM (128 x 2048 x 784 four 6.1, two 6.6, undivided 7.8);
// * two CTAs per SM if each keeps 16 k-blocks: quarters on up to 68 tiles -- 71 found room at once, clusters of four
//   leaving some SMs out, and 72 take two rounds (64 x 2560 x 4096 9.7, in halves 12.4; x 4352 10.3 / 12.8; x 4608 17.3 / 12.8;
//   64 x 2560 x 8192 14.7 / 20.8; 384 x 1024 x 4096 11.0 / 12.8) -- and halves on up to 148 (128 x 4800 x 2048 9.8, undivided 12.1;
//   1000 x 1024 x 4096 15.3 / 21.0), where the rows of both operands start on 32-byte sectors.  Else a row of a box touches five sectors
//   instead of four, the kernel is bound by what L2 delivers, and fewer CTAs are as good or better (1000 x 800 x 3000 halves 19.9,
//   undivided 17.5, but x 3024 15.6 / 17.1; 1000 x 1000 x 2100 15.7 / 13.6; 384 x 1024 x 4100 quarters 16.1, halves 14.4; the largest the
//   other way is 64 x 2512 x 4100, delta, 12.1 / 13.0).  Not in a layer either, which shares the SMs with its neighbours' kernels (16
//   steps of six layers 2048 wide, batch 512, 2490 us undivided, 2910 in halves; 4096 - 1024 at batch 384 2120 in halves, 2160 in quarters);
// * undivided up to 64 k-blocks where the tiles leave no room for more (1000 x 800 x 784 7.9, two 8.3, 128-column tiles 13.5);
// * beyond 64 k-blocks in halves, two CTAs per SM, all the same.
//
// No sum is longer than in the divided form that the shape would otherwise take (the error of a chain grows with its length): one
// CTA where four or two could share the tile has four or two accumulators, and halves have two where quarters could share it.  Relative
// error against 64 bits and time, one sum / in parts / divided: 64 x 64 x 256 2.3e-7 3.5 us / 7.7e-8 3.8 / 7.7e-8 4.3;
// 300 x 1000 x 256 2.3e-7 4.2 / 1.2e-7 4.3 / 1.2e-7 5.7; 1000 x 1000 x 2100 2.2e-6 13.9 / 1.0e-6 13.9 / 1.0e-6 16.9.
int gemm_pick_cluster(int M, int N, int K, int* bn, int* segs, bool layer, bool sectors) {
  *segs = 1;
  if (g_force_bn != 0 || g_force_stages != 0 || g_force_splits != 0 || g_force_persistent >= 0) return 0;
  const long long rows = (M + GEMM_BM - 1) / GEMM_BM;
  const int width = rows * ((N + 63) / 64) <= sm_count() ? 64 : 128;
  const long long tiles = rows * ((N + width - 1) / width);
  const int num_kb = (K + GEMM_BK - 1) / GEMM_BK;
  auto one_each = [&](int c) { return num_kb >= c && tiles * c <= sm_count(); };
  auto two_each = [&](int c) { return tiles * c <= 2 * sm_count() && num_kb >= 16 * c; };
  int c = 0;
  if (width == 64 && num_kb <= 4 && !layer) c = 1, *segs = one_each(4) ? 4 : one_each(2) ? 2 : 1;
  else if ((num_kb >= 16 && tiles <= 8) || (num_kb >= 40 && one_each(8))) c = 8;
  else if (one_each(4) || (sectors && two_each(4) && tiles * 4 <= 2 * sm_count() - 24)) c = 4;
  else if (one_each(2)) c = 2, *segs = two_each(4) ? 2 : 1;
  else if (sectors && two_each(2)) c = 2;
  else if (width == 64 && num_kb <= 64) c = 1, *segs = two_each(2) ? 2 : 1;
  else if (two_each(2)) c = 2;
  // (one tile over a hundred thousand terms: the split through global memory, which a layer has and lp_gemm_bf16 has not,
  // spreads it wider than a cluster can)
  if (c == 0 || (layer && gemm_pick_splits(M, N, K, width) > 2 * c)) return 0;
  *bn = width;
  return c;
}

int gemm_pick_bn(int which, int M, int N, int K, bool allow_pair) {
  if (g_force_bn == 64 || g_force_bn == 128 || g_force_bn == 256) return g_force_bn;
  if (allow_pair && gemm_is_pair(g_force_bn)) return which == 2 ? GEMM_BN_PAIR : g_force_bn;
  if (N <= 64) return 64;
  // tensor-bound shapes: 256 x 256 tiles on SM pairs (code GEMM_BN_PAIR)
  if (allow_pair && M >= 1024 && N >= 1024 && K >= 1024) {
    // forward / delta: a 224-column tile where that fills the last round of SM pairs better (cost =
    // rounds of tiles over the pairs x tile width); G keeps 256 (its update streams 64-column fills)
    if (which != 2 && g_force_bn == 0) {
      const long long pairs = std::max(1, sm_count() / 2), tm = (M + 255) / 256;
      const long long t256 = tm * ((N + 255) / 256), t224 = tm * ((N + 223) / 224);
      if (((t224 + pairs - 1) / pairs) * 224 < ((t256 + pairs - 1) / pairs) * 256) return GEMM_BN_PAIR224;
    }
    return GEMM_BN_PAIR;
  }
  (void)which;
  // 128 x 256 tiles need 96 B/clk of operands per SM instead of 128 B/clk and measured 1250 vs
  // 1130 TFLOP/s on 2048 x 8192 x 8192; they only pay off when the contraction is long and
  // there are enough tiles to fill two CTAs on every SM
  const long long tiles256 = (long long)((M + GEMM_BM - 1) / GEMM_BM) * ((N + 255) / 256);
  if (K >= 1024 && tiles256 >= 2 * kSMs) return 256;
  // (Narrower tiles for small batches were tried: 128 x 64 tiles make a lone forward kernel
  // 35 % faster, but re-read the activations twice as often, and with every stage's kernels
  // sharing L2 and HBM the whole step got 5 % slower.)
  return 128;
}

void gemm_box_dims(int which, int bn, uint32_t boxA[2], uint32_t boxB[2]) {
  const bool a_mn = (which == 2), b_mn = (which != 0);
  boxA[0] = 64; boxA[1] = a_mn ? 64 : GEMM_BM;
  boxB[0] = 64; boxB[1] = b_mn ? 64 : uint32_t(gemm_is_pair(bn) ? gemm_tile_cols(bn) / 2 : bn);   // a pair CTA stages half of the tile's columns
}


// Which contractions exist in a form split over k: forward and delta of a layer, and G of a convolution.
template <int BN, bool A_MN, int MODE>
constexpr bool kHasSplit = A_MN ? BN <= 128 : MODE != EPI_STORE_F32;

template <int BN, bool A_MN, bool B_MN, int MODE>
static cudaError_t launch_one(const CUtensorMap& tmA, const CUtensorMap& tmB, GemmArgs a, cudaStream_t st,
                              const UpdMaps* um) {
  if (a.splits < 1 || a.partial == nullptr) a.splits = 1;
  if (a.splits > 1 && !kHasSplit<BN, A_MN, MODE>) return cudaErrorInvalidValue;
  if (a.wait_limit <= 0) a.wait_limit = LP_WAIT_LIMIT_CYCLES;
  const int num_kb = (a.K + GEMM_BK - 1) / GEMM_BK;
  a.kb_per_split = (num_kb + a.splits - 1) / a.splits;
  const int tiles_m = (a.M + GEMM_BM - 1) / GEMM_BM;
  int tiles_n = (a.N - a.n_begin + BN - 1) / BN;
  if (a.g.kind == GEOM_PIX_K) tiles_n = a.g.n_per_tap * (a.N / a.g.tap_pitch);   // (tap, channel block)
  const long long work = (long long)tiles_m * tiles_n * (a.g.classes > 1 ? a.g.classes : a.splits);
  // BN <= 128: two CTAs per SM (2 x 2 x BN tensor-memory columns); BN = 256: one.
  // Many short tiles (convolutions over large images: thousands of tiles of 9..72 k-blocks) are
  // run by persistent CTAs -- no per-tile launch, barrier and tensor-memory set-up, epilogue
  // overlapped with the next main loop: 64 -> 64 channels at 224 x 224 forward 891 -> 546 us.
  // Few or long tiles keep one tile per CTA with a deeper pipeline: measured on the 8 x 4096
  // workload the persistent form was slower there (step 1.08 vs 0.90 ms), because the fused
  // update epilogue dominates its tiles and a second resident CTA hides more of its latency.
  const int per_sm = BN <= 128 ? 2 : 1;
  const long long slots = (long long)sm_count() * per_sm;
  a.persistent = (work >= 4 * slots && a.kb_per_split <= 96) ? 1 : 0;
  if (g_force_persistent >= 0) a.persistent = g_force_persistent;
  if (a.starve_kb > 0) a.persistent = 0;      // (the starved producer only keeps its ring position for one tile)
  // fused update streamed by TMA: plain geometry, no split-K, tiles at least 128 columns wide
  static const UpdMaps no_maps{};
  a.upd_tma = (MODE == EPI_WGRAD_UPDATE && um != nullptr && a.splits == 1 && BN >= 128 && a.g.kind == GEOM_PLAIN) ? 1 : 0;
  if (!a.upd_tma) um = &no_maps;
  const int stage_bytes = GEMM_A_BYTES + BN * GEMM_BK * 2;
  const int tail = a.upd_tma ? 1024 + UPD_RING_BYTES : 256 + (a.persistent ? EPI_TILE_BYTES : 0);
  const int avail = (per_sm == 2 ? 113 : 227) * 1024 - 1024 - 512 - tail;
  int s = g_force_stages > 0 ? g_force_stages : avail / stage_bytes;
  s = std::max(2, std::min(s, GEMM_MAX_STAGES));
  if (!a.persistent) s = std::max(2, std::min(s, std::max(a.kb_per_split + (a.upd_tma ? BN / 32 : 0), 2)));
  while (s > 2 && size_t(s) * stage_bytes > size_t(227 * 1024 - 1024 - 512 - 1024 - EPI_TILE_BYTES)) --s;
  a.num_stages = s;
  const size_t smem = GemmSmem<BN>::bytes(s, a.persistent != 0, a.upd_tma != 0);
  const int grid = int(a.persistent ? std::min<long long>(work, slots) : work);
  // single-wave launches stream their weights once: request them into L2 well ahead of the pipeline
  a.l2_ahead = (a.g.kind == GEOM_PLAIN && work <= slots && a.kb_per_split >= 8) ? g_l2_ahead : 0;
#define LP_LAUNCH(SPL, PER) \
  launch_chained(gemm_tcgen05_kernel<BN, A_MN, B_MN, MODE, SPL, PER>, grid, GEMM_THREADS, smem, st, 1, tmA, tmB, *um, a, tiles_m, tiles_n, int(work))
  if constexpr (MODE == EPI_WGRAD_UPDATE && BN >= 128) {
    if (a.upd_tma) {
      note_form(a.persistent ? "single streamed persistent" : "single streamed", BN);
      return launch_chained(a.persistent ? gemm_tcgen05_kernel<BN, A_MN, B_MN, MODE, false, true, true> : gemm_tcgen05_kernel<BN, A_MN, B_MN, MODE, false, false, true>,
                            grid, GEMM_THREADS, smem, st, 1, tmA, tmB, *um, a, tiles_m, tiles_n, int(work));
    }
  }
  note_form(a.splits > 1 ? (a.persistent ? "single split persistent" : "single split") : (a.persistent ? "single persistent" : "single"), BN);
  if constexpr (kHasSplit<BN, A_MN, MODE>) {
    if (a.splits > 1) {
      const cudaError_t e = a.persistent ? LP_LAUNCH(true, true) : LP_LAUNCH(true, false);
      if (e != cudaSuccess) return e;
      constexpr int blocks = GEMM_BM * (BN / 4) / 256;      // per tile with one lane
      const int tiles = tiles_m * tiles_n;
      if (a.splits >= 16) return launch_chained(gemm_split_finish_kernel<BN, MODE, 8>, tiles * blocks * 8, 256, 0, st, 1, a, tiles_m, tiles_n);
      return launch_chained(gemm_split_finish_kernel<BN, MODE, 1>, tiles * blocks, 256, 0, st, 1, a, tiles_m, tiles_n);
    }
  }
  return a.persistent ? LP_LAUNCH(false, true) : LP_LAUNCH(false, false);
#undef LP_LAUNCH
}

template <int BN, bool A_MN, bool B_MN, int MODE>
static cudaError_t configure_one() {
  cudaError_t e;
#define LP_ATTR(SPL, PER)                                                                                   \
  if ((e = cudaFuncSetAttribute(gemm_tcgen05_kernel<BN, A_MN, B_MN, MODE, SPL, PER>,                          \
                                cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024)) != cudaSuccess)   \
    return e;
  LP_ATTR(false, false) LP_ATTR(false, true)
  if constexpr (kHasSplit<BN, A_MN, MODE>) { LP_ATTR(true, false) LP_ATTR(true, true) }
#undef LP_ATTR
  if constexpr (MODE == EPI_WGRAD_UPDATE && BN >= 128) {
    if ((e = cudaFuncSetAttribute(gemm_tcgen05_kernel<BN, A_MN, B_MN, MODE, false, false, true>,
                                  cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024)) != cudaSuccess)
      return e;
    if ((e = cudaFuncSetAttribute(gemm_tcgen05_kernel<BN, A_MN, B_MN, MODE, false, true, true>,
                                  cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024)) != cudaSuccess)
      return e;
  }
  return cudaSuccess;
}

// instantiated combinations: (operand majors of the contraction) x (epilogue)
#define LP_FOR_EACH_VARIANT(X, BN)           \
  X(BN, false, false, EPI_FPROP)             \
  X(BN, false, false, EPI_STORE_F32)         \
  X(BN, false, true, EPI_DGRAD)              \
  X(BN, false, true, EPI_DGRAD_UNPOOL)       \
  X(BN, false, true, EPI_STORE_F32)          \
  X(BN, true, true, EPI_STORE_F32)           \
  X(BN, true, true, EPI_WGRAD_UPDATE)

// ---- contraction divided over a cluster ------------------------------------------------------------
template <int BN, bool A_MN, bool B_MN, int MODE>
static cudaError_t launch_cluster(const CUtensorMap& tmA, const CUtensorMap& tmB, GemmArgs a, cudaStream_t st) {
  if (a.wait_limit <= 0) a.wait_limit = LP_WAIT_LIMIT_CYCLES;
  const int tiles_m = (a.M + GEMM_BM - 1) / GEMM_BM, tiles_n = (a.N - a.n_begin + BN - 1) / BN;
  note_form("cluster", BN, a.cluster);
  auto* kernel = gemmc_kernel<BN, A_MN, B_MN, MODE, false, 1>;
  if constexpr (BN == 64) {
    if (a.cluster == 1) kernel = a.segs == 4 ? gemmc_kernel<64, A_MN, B_MN, MODE, true, 4> : a.segs == 2 ? gemmc_kernel<64, A_MN, B_MN, MODE, true, 2> : gemmc_kernel<64, A_MN, B_MN, MODE, true, 1>;
    else if (a.segs == 2) kernel = gemmc_kernel<64, A_MN, B_MN, MODE, false, 2>;
  } else if (a.cluster == 1 || a.segs != 1) {
    return cudaErrorInvalidValue;
  }
  return launch_chained(kernel, dim3(a.cluster, tiles_m * tiles_n), GEMM_THREADS, gemmc_smem_bytes(BN), st, a.cluster, tmA, tmB, a, tiles_m);
}
#define LP_FOR_EACH_CLUSTER_VARIANT(X, BN) \
  X(BN, false, false, EPI_FPROP)           \
  X(BN, false, false, EPI_STORE_F32)       \
  X(BN, false, true, EPI_DGRAD)            \
  X(BN, false, true, EPI_DGRAD_UNPOOL)     \
  X(BN, false, true, EPI_STORE_F32)        \
  X(BN, true, true, EPI_STORE_F32)

// ---- two-CTA (SM pair) kernel ---------------------------------------------------------------
template <bool A_MN, bool B_MN, int MODE, int BN2 = GEMM2_BN>
static cudaError_t launch_pair(const CUtensorMap& tmA, const CUtensorMap& tmB, GemmArgs a, cudaStream_t st, const UpdMaps* um) {
  a.splits = 1;
  if (a.wait_limit <= 0) a.wait_limit = LP_WAIT_LIMIT_CYCLES;
  static const UpdMaps no_maps{};
  a.upd_tma = (MODE == EPI_WGRAD_UPDATE && um != nullptr) ? 1 : 0;
  if (!a.upd_tma) um = &no_maps;
  const int stage_bytes = 32 * 1024;
  const int num_kb = (a.K + GEMM_BK - 1) / GEMM_BK;
  // 3 x 32 KiB: two CTAs per SM, one's epilogue under the other's main loop; 6 where a CTA has its SM to itself anyway,
  // the launch having no more tiles than there are SM pairs (1024 x 4096 x 4096: 37.2 -> 29.1 us)
  const long long all_tiles = (long long)((a.M + 255) / 256) * ((a.N - a.n_begin + BN2 - 1) / BN2);
  const bool alone = all_tiles <= std::max(1, sm_count() / 2);
  int s = g_force_stages > 0 ? g_force_stages : (alone ? 6 : 3);
  s = std::max(2, std::min(std::min(s, GEMM_MAX_STAGES), std::max(num_kb + (a.upd_tma ? GEMM2_BN / 64 : 0), 2)));
  const size_t tail = 1024 + 256 + (a.upd_tma ? 1024 + UPD_RING_BYTES : 0);   // alignment slack, barriers, bf16 staging tile
  while (s > 2 && size_t(s) * stage_bytes + tail > 227 * 1024) --s;
  a.num_stages = s;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * ((a.M + 255) / 256), (a.N - a.n_begin + BN2 - 1) / BN2, 1);
  cfg.blockDim = dim3(GEMM_THREADS, 1, 1);
  cfg.dynamicSmemBytes = size_t(s) * stage_bytes + tail;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if constexpr (MODE == EPI_WGRAD_UPDATE && BN2 == GEMM2_BN) {
    if (a.upd_tma) {
      // Many short tiles (G of a wide layer contracts over the minibatch only): one persistent CTA pair
      // per SM pair, update streamed under the next tile's main loop (8192 x 8192 x 2048: 255 -> 248 us).
      const int tiles_m = (a.M + 255) / 256, tiles_n = (a.N + GEMM2_BN - 1) / GEMM2_BN;
      const int pairs = std::max(1, sm_count() / 2);
      // (with momentum the one-tile form measured faster: 337 against 371 us on 8192 x 8192 x 2048)
      const bool persistent = g_force_persistent >= 0 ? g_force_persistent == 1
                                                      : (tiles_m * tiles_n >= 2 * pairs && num_kb <= 96 && a.mW == nullptr);
      if (persistent && a.starve_kb == 0) {
        cfg.gridDim = dim3(2 * std::min(tiles_m * tiles_n, pairs), 1, 1);
        cfg.blockDim = dim3(GEMM2P_THREADS, 1, 1);
        cfg.dynamicSmemBytes = GEMM2P_SMEM_BYTES;
        // 192 KiB of shared memory divided between operand stages and update-chunk slots
        // (chunk slots are 16 KiB, 32 KiB with momentum: four operand stages leave four / two of them, three leave six / three)
        a.num_stages = g_force_stages > 0 ? std::max(2, std::min(g_force_stages, 5)) : (a.mW != nullptr ? 3 : 4);
        note_form("pair streamed persistent", BN2);
        return cudaLaunchKernelEx(&cfg, gemm2p_g_update_kernel<0>, tmA, tmB, *um, a, tiles_m, tiles_n);
      }
      note_form("pair streamed", BN2, s);
      return cudaLaunchKernelEx(&cfg, gemm2_tcgen05_kernel<A_MN, B_MN, MODE, true>, tmA, tmB, *um, a);
    }
  }
  if constexpr (MODE == EPI_STORE_F32 || (!A_MN && (MODE == EPI_FPROP || MODE == EPI_DGRAD))) {
    // A pair CTA that has its SM to itself walks the tiles with two accumulators (see gemm2q.cuh)
    const int tiles_m = (a.M + 255) / 256, tiles_n = (a.N - a.n_begin + BN2 - 1) / BN2;
    const int pairs = std::max(1, sm_count() / 2);
    // also for the delta contraction of wide fully connected layers (MN-major B: 211 -> 206 us on 2048 x 8192 x 8192
    // in a burst, 252 -> 246 us in a 300-step run; the forward contraction measures the same either way)
    const bool long_delta = MODE == EPI_DGRAD && tiles_m * tiles_n >= 2 * pairs && num_kb >= 32;
    // and for plain fp32 results of at least two tiles per SM pair (4096 x 4096 x 1024: 39.3 -> 35.7 us, 4096^3: 105 -> 100 us)
    const bool many_stores = MODE == EPI_STORE_F32 && tiles_m * tiles_n >= 2 * pairs;
    if (((g_force_persistent == 1 && MODE != EPI_STORE_F32) || long_delta || many_stores) && a.starve_kb == 0 && g_force_persistent != 0 &&
        g_force_stages == 0) {
      cfg.gridDim = dim3(2 * std::min(tiles_m * tiles_n, pairs), 1, 1);
      cfg.blockDim = dim3(GEMM2Q_THREADS, 1, 1);
      cfg.dynamicSmemBytes = GEMM2Q_SMEM_BYTES;
      a.num_stages = GEMM2Q_STAGES;
      note_form("pair persistent", BN2);
      return cudaLaunchKernelEx(&cfg, gemm2q_kernel<A_MN, B_MN, MODE, BN2>, tmA, tmB, a, tiles_m, tiles_n);
    }
  }
  note_form("pair", BN2, s);
  return cudaLaunchKernelEx(&cfg, gemm2_tcgen05_kernel<A_MN, B_MN, MODE, false, BN2>, tmA, tmB, *um, a);
}
template <bool A_MN, bool B_MN, int MODE>
static cudaError_t configure_pair() {
  cudaError_t e = cudaFuncSetAttribute(gemm2_tcgen05_kernel<A_MN, B_MN, MODE, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       227 * 1024);
  if constexpr (MODE == EPI_WGRAD_UPDATE) {
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(gemm2_tcgen05_kernel<A_MN, B_MN, MODE, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  } else if constexpr (!A_MN) {      // forward / delta also exist with 224-column tiles
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(gemm2_tcgen05_kernel<A_MN, B_MN, MODE, false, 224>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(gemm2q_kernel<A_MN, B_MN, MODE, 224>, cudaFuncAttributeMaxDynamicSharedMemorySize, GEMM2Q_SMEM_BYTES);
  }
  if constexpr (MODE != EPI_WGRAD_UPDATE) {
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(gemm2q_kernel<A_MN, B_MN, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, GEMM2Q_SMEM_BYTES);
  }
  return e;
}
#define LP_FOR_EACH_PAIR_VARIANT(X)   \
  X(false, false, EPI_FPROP)          \
  X(false, false, EPI_STORE_F32)      \
  X(false, true, EPI_DGRAD)           \
  X(false, true, EPI_STORE_F32)       \
  X(true, true, EPI_STORE_F32)        \
  X(true, true, EPI_WGRAD_UPDATE)

// ---- halo-tile convolution (3x3, at most 64 channels on both sides) ------------------------------
#define LP_FOR_EACH_HALO_FORM(X, B, M) \
  X(B, M, 1, false) X(B, M, 2, false) X(B, M, 3, false) X(B, M, 4, false) X(B, M, 1, true) X(B, M, 2, true) X(B, M, 3, true) X(B, M, 4, true)
#define LP_FOR_EACH_HALO_VARIANT(X)          \
  LP_FOR_EACH_HALO_FORM(X, false, EPI_FPROP) \
  LP_FOR_EACH_HALO_FORM(X, true, EPI_DGRAD)  \
  LP_FOR_EACH_HALO_FORM(X, true, EPI_DGRAD_UNPOOL)

cudaError_t conv_halo_launch(int which, const CUtensorMap& tmA, const CUtensorMap& tmB, const CUtensorMap& tmO,
                             const GemmArgs& args, cudaStream_t st) {
  const bool b_mn = (which != 0);
  const int tiles = args.g.kind == GEOM_PLAIN ? (args.M + GEMM_BM - 1) / GEMM_BM
                                               : args.g.tiles_w * args.g.tiles_h * (args.M / (args.g.H * args.g.W));
  const int grid = std::min(tiles, sm_count());
  note_form(args.g.kind == GEOM_PLAIN ? "halo plain" : "halo", 64);
  // tiles in turn where a tile's MMAs are few: at most 32 output channels, or a single tap
  const bool turns = args.N <= 32 || args.g.kind == GEOM_PLAIN;
#define LP_TRYH(B, M, S, T)                                                                                    \
  if (b_mn == B && args.mode == M && args.g.last_slices == S && turns == T)                                    \
    return launch_chained(conv_halo_kernel<B, M, S, T>, grid, HALO_THREADS, HALO_SMEM_BYTES, st, 1, tmA, tmB, tmO, args, tiles);
  LP_FOR_EACH_HALO_VARIANT(LP_TRYH)
#undef LP_TRYH
  return cudaErrorInvalidValue;
}

#define LP_FOR_EACH_WIDE_VARIANT(X) X(false, EPI_FPROP) X(true, EPI_DGRAD) X(true, EPI_DGRAD_UNPOOL)
cudaError_t conv_wide_launch(int which, const CUtensorMap& tmA, const CUtensorMap& tmB, const GemmArgs& args, cudaStream_t st) {
  const bool b_mn = (which != 0);
  GemmArgs a = args;
  if (a.wait_limit <= 0) a.wait_limit = LP_WAIT_LIMIT_CYCLES;
  const int tiles = a.g.tiles_w * a.g.tiles_h * (a.M / (a.g.H * a.g.W)), tiles_n = (a.N - a.n_begin + WIDE_BN - 1) / WIDE_BN;
  const int grid = std::min((tiles + 1) / 2 * tiles_n, sm_count());
  note_form("wide halo", WIDE_BN);
#define LP_TRYW(B, M)                                                                                          \
  if (b_mn == B && a.mode == M)                                                                                \
    return launch_chained(conv_wide_kernel<B, M>, grid, WIDE_THREADS, WIDE_SMEM_BYTES, st, 1, tmA, tmB, a, tiles, tiles_n);
  LP_FOR_EACH_WIDE_VARIANT(LP_TRYW)
#undef LP_TRYW
  return cudaErrorInvalidValue;
}

// G of a halo-tile layer: accumulate over 8 x 16 pixel tiles, then add the CTAs' partial sums and
// apply the update (upd.W null: store G only).
cudaError_t conv_halo_g_launch(const CUtensorMap& tmX, const CUtensorMap& tmD, const ConvGeom& g, int batch, float* partial,
                               HaloGUpdate upd, int* status, cudaStream_t st) {
  const int tiles = g.tiles_w * g.tiles_h * batch;
  const int grid = std::min(tiles, sm_count());
  upd.partial = partial;
  upd.n_ctas = grid;
  for (int co0 = 0; co0 < upd.n_out; co0 += 64) {      // one pass per 64 output channels; the stream orders the reuse of `partial`
    note_form("halo G", 64);
    cudaError_t e = launch_chained(conv_halo_g_kernel<0>, grid, GEMM_THREADS, HALOG_SMEM_BYTES, st, 1, tmX, tmD, g, tiles, co0, partial, status);
    if (e != cudaSuccess) return e;
    upd.co0 = co0;
    e = launch_chained(conv_halo_g_update_kernel<0>, HALOG_PART_FLOATS / 32, 256, 0, st, 1, upd);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}
int conv_halo_g_max_ctas() { return sm_count(); }

cudaError_t gemm_configure() {
  cudaError_t e;
  if ((e = cudaFuncSetAttribute(gemm2p_g_update_kernel<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, GEMM2P_SMEM_BYTES)) != cudaSuccess)
    return e;
  if ((e = cudaFuncSetAttribute(conv_halo_g_kernel<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, HALOG_SMEM_BYTES)) != cudaSuccess)
    return e;
#define LP_CFGH(B, M, S, T)                                                                                    \
  if ((e = cudaFuncSetAttribute(conv_halo_kernel<B, M, S, T>, cudaFuncAttributeMaxDynamicSharedMemorySize,           \
                                HALO_SMEM_BYTES)) != cudaSuccess)                                              \
    return e;
  LP_FOR_EACH_HALO_VARIANT(LP_CFGH)
#undef LP_CFGH
#define LP_CFGW(B, M)                                                                                          \
  if ((e = cudaFuncSetAttribute(conv_wide_kernel<B, M>, cudaFuncAttributeMaxDynamicSharedMemorySize,           \
                                WIDE_SMEM_BYTES)) != cudaSuccess)                                              \
    return e;
  LP_FOR_EACH_WIDE_VARIANT(LP_CFGW)
#undef LP_CFGW
#define LP_CFGP(A, B, M) \
  if ((e = configure_pair<A, B, M>()) != cudaSuccess) return e;
  LP_FOR_EACH_PAIR_VARIANT(LP_CFGP)
#undef LP_CFGP
#define LP_CFGC(BN, A, B, M, ONE, SEGS)                                                                        \
  if ((e = cudaFuncSetAttribute(gemmc_kernel<BN, A, B, M, ONE, SEGS>, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                                gemmc_smem_bytes(BN))) != cudaSuccess)                                         \
    return e;
#define LP_CFGC64(BN, A, B, M)                                                                                 \
  LP_CFGC(BN, A, B, M, false, 1) LP_CFGC(BN, A, B, M, false, 2)                                                \
  LP_CFGC(BN, A, B, M, true, 1) LP_CFGC(BN, A, B, M, true, 2) LP_CFGC(BN, A, B, M, true, 4)
#define LP_CFGC128(BN, A, B, M) LP_CFGC(BN, A, B, M, false, 1)
  LP_FOR_EACH_CLUSTER_VARIANT(LP_CFGC64, 64)
  LP_FOR_EACH_CLUSTER_VARIANT(LP_CFGC128, 128)
#undef LP_CFGC128
#undef LP_CFGC64
#undef LP_CFGC
#define LP_CFG(BN, A, B, M) \
  if ((e = configure_one<BN, A, B, M>()) != cudaSuccess) return e;
  LP_FOR_EACH_VARIANT(LP_CFG, 64)
  LP_FOR_EACH_VARIANT(LP_CFG, 128)
  LP_FOR_EACH_VARIANT(LP_CFG, 256)
#undef LP_CFG
  return cudaSuccess;
}

cudaError_t gemm_launch(int which, int bn, const CUtensorMap& tmA, const CUtensorMap& tmB, const GemmArgs& args,
                        cudaStream_t st, const UpdMaps* um) {
  const bool a_mn = (which == 2), b_mn = (which != 0);
  if (gemm_is_pair(bn) && args.g.kind != GEOM_PLAIN) return cudaErrorInvalidValue;
  if (bn == GEMM_BN_PAIR224) {
    if (a_mn) return cudaErrorInvalidValue;
#define LP_TRYP224(A, B, M) \
  if (!A && b_mn == B && args.mode == M) return launch_pair<A, B, M, 224>(tmA, tmB, args, st, nullptr);
    LP_FOR_EACH_PAIR_VARIANT(LP_TRYP224)
#undef LP_TRYP224
    return cudaErrorInvalidValue;
  }
  if (bn == GEMM_BN_PAIR) {
#define LP_TRYP(A, B, M) \
  if (a_mn == A && b_mn == B && args.mode == M) return launch_pair<A, B, M>(tmA, tmB, args, st, um);
    LP_FOR_EACH_PAIR_VARIANT(LP_TRYP)
#undef LP_TRYP
    return cudaErrorInvalidValue;
  }
  if (args.cluster > 0 && args.g.kind == GEOM_PLAIN && args.starve_kb == 0) {
#define LP_TRYC(BN, A, B, M) \
  if (bn == BN && a_mn == A && b_mn == B && args.mode == M) return launch_cluster<BN, A, B, M>(tmA, tmB, args, st);
    LP_FOR_EACH_CLUSTER_VARIANT(LP_TRYC, 64)
    LP_FOR_EACH_CLUSTER_VARIANT(LP_TRYC, 128)
#undef LP_TRYC
    return cudaErrorInvalidValue;
  }
#define LP_TRY(BN, A, B, M) \
  if (bn == BN && a_mn == A && b_mn == B && args.mode == M) return launch_one<BN, A, B, M>(tmA, tmB, args, st, um);
  LP_FOR_EACH_VARIANT(LP_TRY, 64)
  LP_FOR_EACH_VARIANT(LP_TRY, 128)
  LP_FOR_EACH_VARIANT(LP_TRY, 256)
#undef LP_TRY
  return cudaErrorInvalidValue;
}

}  // namespace lp

namespace lp {
cudaError_t gemm_set_tmem_table(int* table) {
  return cudaMemcpyToSymbol(g_tmem_table, &table, sizeof(table));
}
}  // namespace lp

// status block of the stand-alone entry point (handles keep theirs in the workspace)
__device__ int g_gemm_status[lp::STATUS_WORDS] = {};

namespace {
// Per device: the address of g_gemm_status there, and whether the kernels' shared-memory attributes
// have been set on it.  Written once per device under the mutex.
constexpr int kMaxGemmDevices = 64;
std::atomic<int*> g_gemm_status_addr[kMaxGemmDevices];
std::mutex g_gemm_setup_mutex;

int gemm_device_setup(int** status_dev) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxGemmDevices) {
    lp::set_global_error("lp_gemm_bf16: no current CUDA device");
    return LP_ERR_CUDA;
  }
  int* p = g_gemm_status_addr[dev].load(std::memory_order_acquire);
  if (p == nullptr) {
    std::lock_guard<std::mutex> lock(g_gemm_setup_mutex);
    p = g_gemm_status_addr[dev].load(std::memory_order_relaxed);
    if (p == nullptr) {
      void* q = nullptr;
      cudaError_t e = cudaGetSymbolAddress(&q, g_gemm_status);
      if (e == cudaSuccess) e = lp::gemm_configure();
      if (e != cudaSuccess || q == nullptr) {
        lp::set_global_error(std::string("lp_gemm_bf16 set-up: ") + cudaGetErrorString(e));
        return LP_ERR_CUDA;
      }
      p = static_cast<int*>(q);
      g_gemm_status_addr[dev].store(p, std::memory_order_release);
    }
  }
  *status_dev = p;
  return LP_OK;
}

int gemm_standalone(int which, int M, int N, int K, const void* A, int lda, const void* B, int ldb, float* C, int ldc,
                    void* stream, long long wait_limit, int starve_kb) {
  using namespace lp;
  if (which < 0 || which > 2 || M < 1 || N < 1 || K < 1 || !A || !B || !C) return LP_ERR_INVALID_ARG;
  if ((lda & 7) || (ldb & 7) || (ldc & 3)) return LP_ERR_INVALID_ARG;
  int* status_dev = nullptr;
  int rc = gemm_device_setup(&status_dev);
  if (rc != LP_OK) return rc;
  int bn = gemm_pick_bn(which, M, N, K);
  int segs = 1;
  const bool sectors = lda % 16 == 0 && ldb % 16 == 0 && ((reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(B)) & 31) == 0;
  const int cluster = gemm_is_pair(bn) ? 0 : gemm_pick_cluster(M, N, K, &bn, &segs, false, sectors);
  uint32_t boxA[2], boxB[2];
  gemm_box_dims(which, bn, boxA, boxB);
  CUtensorMap tmA, tmB;
  std::string err;
  // A: forward/delta K-major -> rows = M, inner = K; G: stored [K][M] -> inner = M, rows = K
  if (which == 2) rc = make_tmap_bf16_2d(&tmA, A, M, K, lda, boxA[0], boxA[1], &err);
  else            rc = make_tmap_bf16_2d(&tmA, A, K, M, lda, boxA[0], boxA[1], &err);
  if (rc != LP_OK) { set_global_error(err); return rc; }
  // B: forward stored [N][K]; delta and G stored [K][N]
  if (which == 0) rc = make_tmap_bf16_2d(&tmB, B, K, N, ldb, boxB[0], boxB[1], &err);
  else            rc = make_tmap_bf16_2d(&tmB, B, N, K, ldb, boxB[0], boxB[1], &err);
  if (rc != LP_OK) { set_global_error(err); return rc; }
  GemmArgs a{};
  a.M = M; a.N = N; a.K = K;
  a.mode = EPI_STORE_F32;
  a.out = C; a.ld_out = ldc;
  a.status = status_dev;
  a.wait_limit = wait_limit;
  a.starve_kb = starve_kb;
  a.cluster = cluster;
  a.segs = segs;
  cudaError_t e = gemm_launch(which, bn, tmA, tmB, a, static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) { set_global_error(std::string("lp_gemm_bf16 launch: ") + cudaGetErrorString(e)); return LP_ERR_CUDA; }
  return LP_OK;
}
}  // namespace

// ---------------------------------------------------------------------------
extern "C" int lp_gemm_bf16(int which, int M, int N, int K, const void* A, int lda, const void* B, int ldb,
                            float* C, int ldc, void* stream) {
  return gemm_standalone(which, M, N, K, A, lda, B, ldb, C, ldc, stream, 0, 0);
}

extern "C" const char* lp_debug_last_contraction(void) { return lp::gemm_last_contraction(); }

extern "C" int lp_gemm_status(int* detail) {
  int* status_dev = nullptr;
  int rc = gemm_device_setup(&status_dev);
  if (rc != LP_OK) return rc;
  int st[lp::STATUS_WORDS] = {};
  const int zero[lp::STATUS_WORDS] = {};
  if (cudaDeviceSynchronize() != cudaSuccess || cudaMemcpy(st, status_dev, sizeof st, cudaMemcpyDeviceToHost) != cudaSuccess ||
      cudaMemcpy(status_dev, zero, sizeof zero, cudaMemcpyHostToDevice) != cudaSuccess) {
    lp::set_global_error("lp_gemm_status: a CUDA call failed");
    return LP_ERR_CUDA;
  }
  if (detail) *detail = st[lp::STATUS_CODE];
  if (st[lp::STATUS_CODE] != 0) {
    lp::set_global_error("lp_gemm_bf16: " + lp::expired_text(st));
    return LP_ERR_TIMEOUT;
  }
  return LP_OK;
}

extern "C" int lp_debug_gemm_starved(int M, int N, int K, const void* A, int lda, const void* B, int ldb, float* C,
                                     int ldc, long long limit_cycles, void* stream) {
  if (limit_cycles < 1000 || limit_cycles > 2000000000ll || K <= lp::GEMM_BK) return LP_ERR_INVALID_ARG;
  return gemm_standalone(0, M, N, K, A, lda, B, ldb, C, ldc, stream, limit_cycles, 1);
}
