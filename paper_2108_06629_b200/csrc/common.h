// Internal declarations shared by the host-side translation units.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <string>
#include <utility>
#include <vector>

#include "../../include/layerpipe.h"
#include "wait_codes.h"

namespace lp {

// Streaming multiprocessors of a B200.  Sizes and rules that must come out the same with and without a device in the
// process (workspace, splits, kernel forms of a layer) use this number; grids of launches ask the device.
constexpr int kSMs = 148;

// ---- launches -----------------------------------------------------------------
// Kernels of a stream follow one another at once: the launch carries the programmatic-serialisation attribute, so the
// next kernel's blocks may start when every block of the one before has called launch_next() or ended, and
// launch_wait() in front of their first access to global memory holds them until that one has completed and its writes are
// visible.  Behind a kernel that calls launch_next() their set-up (barriers, tensor memory, descriptors) runs under its tail; behind the others,
// the tile kernels among them, it is the launch's own latency that is saved.  Every thread block executes the wait, so
// completion stays transitive along a stream whatever the launches in between did.
// Where an event wait stands between two launches the attribute has no effect.  Measured on a chain of one-block kernels: 1.9 us
// from the end of a kernel to the start of the next one, 0.54 us with the attribute; the launch call itself 2.9 -> 2.4 us.
template <class... KArgs, class... Args>
inline cudaError_t launch_chained(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, int cluster, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}
// Holds until the kernel before this one in the stream has completed (returns at once in a launch without the attribute).  What that
// kernel writes changes while this one runs: no __restrict__ on parameters and no read-only loads, which the compiler may move in front.
__device__ __forceinline__ void launch_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// The next kernel of the stream may start its blocks once every block of this one has said so or has ended.  Said by the
// kernels of short chains only (cluster contractions, loss, column sums), once a block has asked for its last operands.  Blocks that
// wait take room from other streams: with the tile kernels saying it too, 16 steps of the small VGG took 4370 us
// (4160 without, 4260 with plain launches) and nothing was faster for it.
__device__ __forceinline__ void launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ---- lp_api.cu --------------------------------------------------------------
// Error text of calls that have no handle: what lp_last_error(NULL) returns on this thread.
void set_global_error(const std::string& msg);
// What a status block says: which role of which kernel gave up first, and where it stood.
inline std::string expired_text(const int* st) {
  const int code = st[STATUS_CODE];
  return std::string("a bounded device-side wait expired: ") + wait_code_role(code) + " of the " + wait_code_name(code) + " kernel (status " +
         std::to_string(code) + "; CTA " + std::to_string(st[STATUS_CTA]) + ", tile " + std::to_string(st[STATUS_TILE]) + ", step " +
         std::to_string(st[STATUS_STEP]) + ")";
}

// ---- gemm.cu ---------------------------------------------------------------
// Encode a 2-D bf16 tensor map (128-byte swizzle, zero fill out of bounds).
// inner/outer are the logical extents in elements, pitch_elems the row pitch.
int make_tmap_bf16_2d(CUtensorMap* out, const void* base, uint64_t inner, uint64_t outer,
                      uint64_t pitch_elems, uint32_t box_inner, uint32_t box_outer, std::string* err);

int make_tmap_bf16_nhwc(CUtensorMap* out, const void* base, uint64_t C, uint64_t W, uint64_t H, uint64_t N,
                        uint64_t pitch_c, uint32_t bw, uint32_t bh, uint32_t bn, std::string* err, uint32_t step = 1);

// fp32 (elem_bytes 4) or bf16 (2) row-major tensor moved in boxes of 32 columns x box_outer rows
// (the streamed tiles of the fused update).
int make_tmap_rows32(CUtensorMap* out, const void* base, int elem_bytes, uint64_t inner, uint64_t outer,
                     uint64_t pitch_elems, uint32_t box_outer, std::string* err);

struct GemmArgs;
struct UpdMaps;
constexpr int GEMM_BN_PAIR = 512;   // tile code: 256 x 256 tile computed by a pair of CTAs (cta_group::2)
constexpr int GEMM_BN_PAIR224 = 448;   // tile code: 256 x 224 tile on a pair of CTAs (forward / delta only)
inline bool gemm_is_pair(int bn) { return bn == GEMM_BN_PAIR || bn == GEMM_BN_PAIR224; }
inline int gemm_tile_cols(int bn) { return gemm_is_pair(bn) ? bn / 2 : bn; }   // output columns of one tile
// which: 0 forward (A,B K-major), 1 delta (B MN-major), 2 G (A,B MN-major).
// Tile width BN is chosen from N and the box sizes of tmA/tmB must match it
// (see gemm_box_dims).
int gemm_pick_bn(int which, int M, int N, int K, bool allow_pair = true);
void gemm_box_dims(int which, int bn, uint32_t boxA[2], uint32_t boxB[2]);
// um (EPI_WGRAD_UPDATE only): tensor maps of the master, momentum and destination ring slot; when
// given, and the launch qualifies, the update's tiles are streamed by TMA.
cudaError_t gemm_launch(int which, int bn, const CUtensorMap& tmA, const CUtensorMap& tmB,
                        const GemmArgs& args, cudaStream_t stream, const UpdMaps* um = nullptr);
// 3x3 convolution forward (which = 0) / delta (which = 1) with at most 64 channels on both sides:
// tmA = NHWC tensor map with a 64 x 10 x 18 x 1 box, tmB = the layer's weight map (64 x 64 boxes);
// args.g describes 8 x 16 pixel tiles (lw = 3, lh = 4).  tmO (forward only; any valid map otherwise): the
// NHWC output with a 64 x 8 x 16 x 1 box, written by TMA stores.  With plain geometry (which = 0 only) the
// call is a forward GEMM with K <= 64 and N <= 64: tmA and tmO are 2-D maps with 64 x 128 boxes.
cudaError_t conv_halo_launch(int which, const CUtensorMap& tmA, const CUtensorMap& tmB, const CUtensorMap& tmO,
                             const GemmArgs& args, cudaStream_t stream);
// The same with more than 64 channels on a side (conv_wide.cuh); tmB with boxes of 128 output columns.
cudaError_t conv_wide_launch(int which, const CUtensorMap& tmA, const CUtensorMap& tmB, const GemmArgs& args, cudaStream_t stream);
struct ConvGeom;
struct HaloGUpdate;
// G (+ fused update) of a halo-tile layer: tmX = the activations with the 64 x 10 x 18 x 1 halo box,
// tmD = delta with a 64 x 8 x 16 x 1 box; partial: conv_halo_g_max_ctas() x 5 x 128 x 64 floats.
int conv_halo_g_max_ctas();
const char* gemm_last_contraction();   // see lp_debug_last_contraction
cudaError_t gemm_configure();   // opt in to large dynamic shared memory; call once per process
void gemm_set_tuning(int bn, int stages, int splits);   // 0 = automatic
int gemm_pick_splits(int M, int N, int K, int bn);
// CTAs of a cluster that share one tile's contraction (GemmArgs::cluster) and, where that is not 0, the tile width
// (layer: the epilogue is that of a layer, and there is scratch for a contraction split through global memory, which may be the better one);
// sectors: the rows of both operands start on 32-byte sectors, and the launch has the GPU to itself; *segs: accumulators of
// each of them (GemmArgs::segs)
int gemm_pick_cluster(int M, int N, int K, int* bn, int* segs, bool layer, bool sectors);

// ---- planner.cpp ------------------------------------------------------------
struct PlanResult {
  std::vector<int> stage, delay;
  std::vector<int> piece_stage;          // [2*L]
  std::vector<long long> piece_amount;   // [2*L]
  int used = 0;
  long long Tp = 0;
  int rounds = 0;
};
int plan_layers(const lp_layer* layers, int L, int batch, int Np, PlanResult* out);
int layer_macs(const lp_layer& y, int batch, long long* macs);   // the planner's cost of one contraction of the layer

// ---- elementwise.cu ---------------------------------------------------------
cudaError_t launch_cast_stash(const void* batch, int input_is_bf16, const int* labels, __nv_bfloat16* x0,
                              int* labels_copy, int rows, int B, int n_in, int ld, cudaStream_t stream);
cudaError_t launch_cast_patch3x3(const void* batch, int input_is_bf16, const int* labels, __nv_bfloat16* x0,
                                 int* labels_copy, int B, int H, int W, int C, int ld, cudaStream_t stream);
// The same for any filter, stride and padding (R*S*C <= 128): one row per OUTPUT pixel, column (r*S + s)*C + ch.
cudaError_t launch_cast_patch_general(const void* batch, int input_is_bf16, const int* labels, __nv_bfloat16* x0,
                                      int* labels_copy, int B, int H, int W, int C, int R, int S, int stride, int pad,
                                      int Ho, int Wo, int ld, cudaStream_t stream);
// diagnosis: the per-SM tensor-memory table (160 x 16 ints of device memory, zeroed) that the kernels keep, or null
cudaError_t gemm_set_tmem_table(int* table);
// one thread writes `value` to *flag (mapped host memory): the progress mark after a task
cudaError_t launch_trace_mark(unsigned* flag, unsigned value, cudaStream_t stream);
// ticket: count of finished blocks, zero between launches
cudaError_t launch_softmax_xent(const float* zL, int ldz, const int* labels, __nv_bfloat16* delta, int ldd, float* row_loss,
                                unsigned* ticket, float* loss_out, int B, int C, int* status, cudaStream_t stream);
// Value of a device status word that does not come from a bounded wait (those are in wait_codes.h).
constexpr int LP_STATUS_BAD_LABEL = 64;   // a label outside [0, classes) reached the loss kernel
struct UpdateArgs {
  const float* dW;      // [out][ldw] fp32 (pad lanes zero)
  float* W;             // master [out][ldw]
  float* mW;            // momentum or null
  __nv_bfloat16* ring;  // bf16 slot that receives RN(W)
  long long n_elems;    // out * ldw (multiple of 8)
  const __nv_bfloat16* delta;  // [rows][ldd]: bias gradient = column sums (null: no bias)
  int rows, ldd, n_out;
  float* b;             // master bias
  float* mb;            // bias momentum or null
  float* db;            // bias gradient out
  float* bring;         // fp32 bias slot that receives b
  float lr, mu;
};
// Interleaved partial sums of a bias gradient (row r belongs to sum r mod BIAS_LANES; the sums are then added in order):
// the same in the update kernel and in the G kernel that does the bias as well.  (Four sums of two-byte loads kept that kernel's
// epilogue waiting: 16 steps of the ragged GELU MLP at batch 100, 634 us; eight sums of 16-byte loads 622.)
constexpr int BIAS_LANES = 8;
cudaError_t launch_sgd_update(const UpdateArgs& a, cudaStream_t stream);
// 2x2 stride-2 max pool of an NHWC bf16 tensor (C a multiple of 8); idx = position of the first
// maximum in (dh, dw) row-major order.
cudaError_t launch_maxpool2(const __nv_bfloat16* a, __nv_bfloat16* pooled, unsigned char* idx, int B, int H, int W,
                            int C, cudaStream_t stream);
// Bias gradient (column sums of the [rows][ld] bf16 matrix x, ld a multiple of 8, rows 16-byte aligned) and bias update of a
// layer with more than 512 rows; up to that the single pass inside launch_sgd_update or the G kernel does it.
// partial: colsum_chunks x 64 floats per 64 columns; counter: one word per 64 columns, zero between launches.
struct BiasUpdate {
  float *b, *mb, *db, *bring;   // master, momentum (may be null), gradient out, slot that receives b
  float lr, mu;
};
// About four blocks per SM, but no fewer than 256 rows to a block (its fixed cost is a tail of two block-wide sums).
inline int colsum_chunk_rows(int rows, int n_cols) {
  const int want = std::max(1, 4 * kSMs / ((n_cols + 63) / 64));
  return std::max(256, ((rows + want - 1) / want + 31) / 32 * 32);
}
inline int colsum_chunks(int rows, int n_cols) {
  const int c = colsum_chunk_rows(rows, n_cols);
  return rows > 512 ? (rows + c - 1) / c : 0;
}
cudaError_t launch_colsum_bias(const __nv_bfloat16* x, int rows, int ld, int n_cols, float* partial, unsigned* counter,
                               const BiasUpdate& u, cudaStream_t stream);
cudaError_t launch_round_to_bf16(const float* src, __nv_bfloat16* dst, long long n_elems, cudaStream_t stream);

}  // namespace lp
