// HBM-bound kernels of the training step: input cast + stash, softmax cross-entropy with
// delta^L, and the fused SGD update (Eq. 6) that also refreshes the bf16 weight-ring slot.
#include <atomic>
#include <cstdio>
#include <mutex>

#include "common.h"

namespace lp {

__global__ void trace_mark_kernel(unsigned* flag, unsigned value) {
  *reinterpret_cast<volatile unsigned*>(flag) = value;
  __threadfence_system();
}
cudaError_t launch_trace_mark(unsigned* flag, unsigned value, cudaStream_t stream) {
  trace_mark_kernel<<<1, 1, 0, stream>>>(flag, value);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// a^0 = RN_bf16(batch) into the first layer's activation-stash slot; labels are copied
// into the library's label ring so that the caller may reuse its buffers.
__global__ void cast_stash_kernel(const void* batch, int input_is_bf16,
                                  const int* labels, __nv_bfloat16* x0,
                                  int* labels_copy, int rows, int B, int n_in, int ld) {
  launch_wait();
  const long long groups_per_row = ld / 8;
  const long long total = (long long)rows * groups_per_row;
  for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < total;
       g += (long long)gridDim.x * blockDim.x) {
    const int row = int(g / groups_per_row);
    const int c0 = int(g % groups_per_row) * 8;
    float v[8];
    if (input_is_bf16) {
      const __nv_bfloat16* src = reinterpret_cast<const __nv_bfloat16*>(batch) + (long long)row * n_in;
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = (c0 + j < n_in) ? __bfloat162float(src[c0 + j]) : 0.f;
    } else {
      const float* src = reinterpret_cast<const float*>(batch) + (long long)row * n_in;
      if ((n_in & 3) == 0 && c0 + 8 <= n_in) {
        const float4 a = *reinterpret_cast<const float4*>(src + c0);
        const float4 b = *reinterpret_cast<const float4*>(src + c0 + 4);
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
      } else {
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = (c0 + j < n_in) ? src[c0 + j] : 0.f;
      }
    }
    __nv_bfloat162 p0 = __floats2bfloat162_rn(v[0], v[1]);
    __nv_bfloat162 p1 = __floats2bfloat162_rn(v[2], v[3]);
    __nv_bfloat162 p2 = __floats2bfloat162_rn(v[4], v[5]);
    __nv_bfloat162 p3 = __floats2bfloat162_rn(v[6], v[7]);
    uint4 o;
    o.x = *reinterpret_cast<uint32_t*>(&p0);
    o.y = *reinterpret_cast<uint32_t*>(&p1);
    o.z = *reinterpret_cast<uint32_t*>(&p2);
    o.w = *reinterpret_cast<uint32_t*>(&p3);
    *reinterpret_cast<uint4*>(x0 + (long long)row * ld + c0) = o;
  }
  if (blockIdx.x == 0) {
    for (int i = threadIdx.x; i < B; i += blockDim.x) labels_copy[i] = labels[i];
  }
}

cudaError_t launch_cast_stash(const void* batch, int input_is_bf16, const int* labels, __nv_bfloat16* x0,
                              int* labels_copy, int rows, int B, int n_in, int ld, cudaStream_t stream) {
  const long long total = (long long)rows * (ld / 8);
  int blocks = int(std::min<long long>((total + 255) / 256, kSMs * 8));
  if (blocks < 1) blocks = 1;
  return launch_chained(cast_stash_kernel, blocks, 256, 0, stream, 1, batch, input_is_bf16, labels, x0, labels_copy, rows, B, n_in, ld);
}

// ---------------------------------------------------------------------------
// First convolution layer with very few input channels (an RGB image): a^0 is stashed as the
// matrix of 3x3 patches, one row per output pixel, column (r*3 + s)*C + ch = the input at
// (h + r - 1, w + s - 1, ch) or zero outside the image, padded with zero columns to `ld`.  The
// layer's contractions (Eq. 1 and Eq. 5 written for a convolution) then run as plain GEMMs over
// 9*C columns instead of nine taps of a 64-wide k-block that would be 95 % padding.
// One thread per output pixel; C is a template parameter so that the 9*C gathered values stay in
// registers and the column arithmetic folds at compile time.
template <int C>
__global__ void cast_patch3x3_kernel(const void* batch, int input_is_bf16,
                                     const int* labels, __nv_bfloat16* x0,
                                     int* labels_copy, int B, int H, int W) {
  constexpr int LD = (9 * C + 7) / 8 * 8;
  launch_wait();
  const int total = B * H * W;
  for (int pix = blockIdx.x * blockDim.x + threadIdx.x; pix < total; pix += gridDim.x * blockDim.x) {
    const int w = pix % W;
    const int h = (pix / W) % H;
    float v[LD];
#pragma unroll
    for (int k = 0; k < LD; ++k) v[k] = 0.f;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const int hh = h + r - 1;
      if (hh < 0 || hh >= H) continue;
#pragma unroll
      for (int s = 0; s < 3; ++s) {
        const int ww = w + s - 1;
        if (ww < 0 || ww >= W) continue;
        const long long idx = ((long long)pix + (r - 1) * W + (s - 1)) * C;
#pragma unroll
        for (int ch = 0; ch < C; ++ch)
          v[(r * 3 + s) * C + ch] = input_is_bf16 ? __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(batch)[idx + ch])
                                                  : reinterpret_cast<const float*>(batch)[idx + ch];
      }
    }
    uint4* dst = reinterpret_cast<uint4*>(x0 + (long long)pix * LD);
#pragma unroll
    for (int g = 0; g < LD / 8; ++g) {
      __nv_bfloat162 p0 = __floats2bfloat162_rn(v[8 * g + 0], v[8 * g + 1]);
      __nv_bfloat162 p1 = __floats2bfloat162_rn(v[8 * g + 2], v[8 * g + 3]);
      __nv_bfloat162 p2 = __floats2bfloat162_rn(v[8 * g + 4], v[8 * g + 5]);
      __nv_bfloat162 p3 = __floats2bfloat162_rn(v[8 * g + 6], v[8 * g + 7]);
      uint4 o;
      o.x = *reinterpret_cast<uint32_t*>(&p0);
      o.y = *reinterpret_cast<uint32_t*>(&p1);
      o.z = *reinterpret_cast<uint32_t*>(&p2);
      o.w = *reinterpret_cast<uint32_t*>(&p3);
      dst[g] = o;
    }
  }
  if (blockIdx.x == 0) {
    for (int i = threadIdx.x; i < B; i += blockDim.x) labels_copy[i] = labels[i];
  }
}

cudaError_t launch_cast_patch3x3(const void* batch, int input_is_bf16, const int* labels, __nv_bfloat16* x0,
                                 int* labels_copy, int B, int H, int W, int C, int ld, cudaStream_t stream) {
  const long long total = (long long)B * H * W;
  if (C < 1 || C > 7 || ld != (9 * C + 7) / 8 * 8 || total >= (1ll << 31)) return cudaErrorInvalidValue;
  int blocks = int(std::min<long long>((total + 255) / 256, kSMs * 8));
  if (blocks < 1) blocks = 1;
#define LP_PATCH_CASE(c)                                                                                        \
  case c: return launch_chained(cast_patch3x3_kernel<c>, blocks, 256, 0, stream, 1, batch, input_is_bf16, labels, x0, labels_copy, B, H, W);
  switch (C) {
    LP_PATCH_CASE(1) LP_PATCH_CASE(2) LP_PATCH_CASE(3) LP_PATCH_CASE(4) LP_PATCH_CASE(5) LP_PATCH_CASE(6) LP_PATCH_CASE(7)
  }
#undef LP_PATCH_CASE
  return cudaErrorInvalidValue;
}

// General filters / strides.  A block writes the patch rows of PATCH_PIX output pixels of one image row: it stages the R
// input rows that they touch (zeros outside the image) in shared memory as bf16, in runs of whole pixels -- a tap row of
// a patch, S * C values, is then contiguous there -- and a thread builds 8 columns (one 16-byte store) from two-byte
// shared reads through a table of column offsets.  32 x 224 x 224 x 3, 5x5 stride 2: 128 us when every value was fetched from
// global memory behind divisions, 54 us now with cold caches (84 MB: 13 us at the measured copy rate; the two-byte
// shared reads bound it).
constexpr int PATCH_PIX = 64;
constexpr int PATCH_COLS_MAX = 128;
inline int patch_span(int S, int stride) { return (PATCH_PIX - 1) * stride + S; }     // input pixels of one staged row
__global__ void __launch_bounds__(256)
cast_patch_general_kernel(const void* batch, int input_is_bf16, const int* labels,
                          __nv_bfloat16* x0, int* labels_copy, int B, int H, int W, int C, int R, int S,
                          int stride, int pad, int Ho, int Wo, int ld, int span, int segs) {
  extern __shared__ __nv_bfloat16 rows[];                      // [R][span][C]
  __shared__ short col_off[PATCH_COLS_MAX];                    // column -> offset in `rows` for output pixel 0, -1: padding column
  const int seg = int(blockIdx.x) % segs, ho = (int(blockIdx.x) / segs) % Ho, b = int(blockIdx.x) / (segs * Ho);
  const int wo0 = seg * PATCH_PIX, n_pix = min(PATCH_PIX, Wo - wo0);
  for (int c = threadIdx.x; c < ld; c += blockDim.x) {
    const int tap = c / C;
    col_off[c] = c < R * S * C ? short((tap / S) * span * C + (tap % S) * C + c % C) : short(-1);
  }
  const int w0 = wo0 * stride - pad, row_vals = span * C;
  launch_wait();
  for (int i = threadIdx.x; i < R * row_vals; i += blockDim.x) {
    const int r = i / row_vals, q = i - r * row_vals;
    const int hh = ho * stride - pad + r, x = w0 * C + q;      // x: position in the image row, in values
    __nv_bfloat16 v = __float2bfloat16_rn(0.f);
    if (hh >= 0 && hh < H && x >= 0 && x < W * C) {
      const long long idx = ((long long)b * H + hh) * W * C + x;
      v = input_is_bf16 ? reinterpret_cast<const __nv_bfloat16*>(batch)[idx] : __float2bfloat16_rn(reinterpret_cast<const float*>(batch)[idx]);
    }
    rows[i] = v;
  }
  __syncthreads();
  const int groups = ld / 8;
  __nv_bfloat16* dst = x0 + (((long long)b * Ho + ho) * Wo + wo0) * ld;
  const unsigned short* raw = reinterpret_cast<const unsigned short*>(rows);
  for (int t = threadIdx.x; t < n_pix * groups; t += blockDim.x) {
    const int pix = t / groups, g = t - pix * groups;
    const int base = pix * stride * C;
    uint32_t w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int o0 = col_off[g * 8 + 2 * k], o1 = col_off[g * 8 + 2 * k + 1];
      const uint32_t lo = o0 >= 0 ? raw[base + o0] : 0u, hi = o1 >= 0 ? raw[base + o1] : 0u;
      w[k] = lo | (hi << 16);
    }
    *reinterpret_cast<uint4*>(dst + (long long)t * 8) = make_uint4(w[0], w[1], w[2], w[3]);
  }
  if (blockIdx.x == 0) {
    for (int i = threadIdx.x; i < B; i += blockDim.x) labels_copy[i] = labels[i];
  }
}

cudaError_t launch_cast_patch_general(const void* batch, int input_is_bf16, const int* labels, __nv_bfloat16* x0,
                                      int* labels_copy, int B, int H, int W, int C, int R, int S, int stride, int pad,
                                      int Ho, int Wo, int ld, cudaStream_t stream) {
  const int span = patch_span(S, stride), segs = (Wo + PATCH_PIX - 1) / PATCH_PIX;
  const long long blocks = (long long)B * Ho * segs;
  const size_t smem = size_t(R) * span * C * 2;
  // (filters up to 7x7, stride up to 2, at most 8 channels: 15 KiB)
  if (C < 1 || R * S * C > ld || (ld & 7) || ld > PATCH_COLS_MAX || smem > 48 * 1024 || blocks >= (1ll << 31)) return cudaErrorInvalidValue;
  return launch_chained(cast_patch_general_kernel, int(blocks), 256, smem, stream, 1, batch, input_is_bf16, labels, x0, labels_copy, B, H, W, C,
                        R, S, stride, pad, Ho, Wo, ld, span, segs);
}

// ---------------------------------------------------------------------------
// p = softmax(z^L), delta^L = RN((p - onehot)/B), row loss.  A row belongs to TPR threads (eight, a warp, or the block for
// wide rows), which keep its logits and exponentials in registers: the logits are read once, one exponential per element, 4
// bytes per class in and 2 out.  What bounds it beside memory is the instructions of an element, so there is no test per
// element: lanes past C hold -inf, and the label's owner overwrites its element.  Time of the static call, its
// inputs in L2 or not as 40 calls in a row leave them, before (a comparison per element, 8-byte loads, three or four rows to a
// warp of 72 registers, the counter cleared by a launch in front) and now: 8192 x 1000 22.6 -> 13.3 us, 16384 x 1000 35.2 -> 21.5,
// 16384 x 4000 266 -> 104, 1000 x 1500 20.5 -> 6.0.  (A look-ahead of one row in registers, 128 a thread: 18.4 for the first.)
// VEC: consecutive classes of a thread, 4 or 2 where pitches and addresses allow accesses of that width.
// The mean of the row losses, in a fixed order: by the last block to finish where the caller has a counter for that (a
// trainer), by the block itself where it is the only one, else by a launch of its own (softmax_xent_mean_kernel).
constexpr int XENT_THREADS = 256;

template <int TPR>
__device__ __forceinline__ float row_reduce(float v, float* sh, bool is_max) {
#pragma unroll
  for (int o = TPR < 32 ? TPR / 2 : 16; o > 0; o >>= 1) {
    const float other = __shfl_xor_sync(0xffffffffu, v, o);
    v = is_max ? fmaxf(v, other) : v + other;
  }
  if (TPR <= 32) return v;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  float r = sh[0];
#pragma unroll
  for (int i = 1; i < TPR / 32; ++i) r = is_max ? fmaxf(r, sh[i]) : r + sh[i];
  return r;
}

// Mean of B row losses by the block, in one order whatever the block's size, so that a trainer's loss and the static call's are the
// same bits: sum t of XENT_SUMS takes rows t, t + XENT_SUMS, ... in that order, 32 neighbouring sums are added as a tree, the 32 results in order.
constexpr int XENT_SUMS = 1024;
template <int THREADS>
__device__ __forceinline__ void row_loss_mean(const float* row_loss, float* loss_out, int B, float* sh) {
  constexpr int PER = XENT_SUMS / THREADS;            // sums of a thread
  if (PER > 1 && B <= THREADS) {                      // (the other sums are empty: the same bits)
    const float sum = row_reduce<THREADS>(int(threadIdx.x) < B ? __ldcg(row_loss + threadIdx.x) : 0.f, sh, false);
    if (threadIdx.x == 0) *loss_out = sum * (1.0f / float(B));
    return;
  }
  float acc[PER] = {};
#pragma unroll 8
  for (int i = threadIdx.x; i < B; i += XENT_SUMS)
#pragma unroll
    for (int k = 0; k < PER; ++k)
      if (PER == 1 || i + k * THREADS < B) acc[k] += __ldcg(row_loss + i + k * THREADS);
#pragma unroll
  for (int k = 0; k < PER; ++k) acc[k] = row_reduce<32>(acc[k], nullptr, false);
  __syncthreads();
#pragma unroll
  for (int k = 0; k < PER; ++k)
    if ((threadIdx.x & 31) == 0) sh[k * (THREADS / 32) + int(threadIdx.x >> 5)] = acc[k];
  __syncthreads();
  if (threadIdx.x == 0) {
    float sum = sh[0];
#pragma unroll
    for (int i = 1; i < XENT_SUMS / 32; ++i) sum += sh[i];
    *loss_out = sum * (1.0f / float(B));
  }
}
__global__ void __launch_bounds__(XENT_SUMS) softmax_xent_mean_kernel(const float* row_loss, float* loss_out, int B) {
  __shared__ float sh[XENT_SUMS / 32];
  launch_wait();
  row_loss_mean<XENT_SUMS>(row_loss, loss_out, B, sh);
}

// N = classes that a thread keeps in registers; what lies beyond TPR * N goes in several sweeps over memory
template <int TPR, int VEC, int N>
__global__ void __launch_bounds__(XENT_THREADS, 4)
softmax_xent_kernel(const float* zL, int ldz, const int* labels, __nv_bfloat16* delta, int ldd,
                    float* row_loss, unsigned* ticket, float* loss_out, int B, int C, int* status) {
  constexpr int ROWS = XENT_THREADS / TPR;            // rows of a block
  __shared__ float sh[XENT_SUMS / 32];
  __shared__ bool last;
  const int t = int(threadIdx.x) % TPR;
  const float invB = 1.0f / float(B);
  const int Cpad = (C + 7) & ~7;
  const bool wide = C > TPR * N;
  // position k of thread t is class (k / VEC) * TPR * VEC + t * VEC + k % VEC
  auto cls = [&](int k) { return (k / VEC) * (TPR * VEC) + t * VEC + k % VEC; };
  launch_wait();
  for (int first = blockIdx.x * ROWS; first < B; first += int(gridDim.x) * ROWS) {
    const bool mine = first + int(threadIdx.x) / TPR < B;       // (the last rows' warps keep together: they shuffle)
    const int row = mine ? first + int(threadIdx.x) / TPR : B - 1;
    const float* z = zL + (long long)row * ldz;
    __nv_bfloat16* d = delta + (long long)row * ldd;
    float v[N];
    float mx = -INFINITY, s = 0.f;
#pragma unroll
    for (int k = 0; k < N; k += VEC) {
      const int c = cls(k);
      if (VEC == 4 && c + 3 < C) {
        const float4 w = *reinterpret_cast<const float4*>(z + c);
        v[k] = w.x; v[k + VEC / 4] = w.y; v[k + VEC / 2] = w.z; v[k + VEC - 1] = w.w;
      } else if (VEC == 2 && c + 1 < C) {
        const float2 w = *reinterpret_cast<const float2*>(z + c);
        v[k] = w.x; v[k + VEC - 1] = w.y;
      } else {
#pragma unroll
        for (int e = 0; e < VEC; ++e) v[k + e] = c + e < C ? z[c + e] : -INFINITY;
      }
    }
    const int y = labels[row];
#pragma unroll
    for (int k = 0; k < N; ++k) mx = fmaxf(mx, v[k]);
    if (wide) for (int c = TPR * N + t; c < C; c += TPR) mx = fmaxf(mx, z[c]);
    mx = row_reduce<TPR>(mx, sh, true);
#pragma unroll
    for (int k = 0; k < N; ++k) {
      v[k] = expf(v[k] - mx);                         // (0 in the lanes past C)
      s += v[k];
    }
    if (wide) for (int c = TPR * N + t; c < C; c += TPR) s += expf(z[c] - mx);
    s = row_reduce<TPR>(s, sh, false);
    // Every class as if it were not the label, whose owner then overwrites its element: no comparison per element.
    const float inv_s = 1.0f / s;
#pragma unroll
    for (int k = 0; k < N; k += VEC) {
      const int c = cls(k);
      if (c >= Cpad || !mine) continue;
      float o[VEC];
#pragma unroll
      for (int e = 0; e < VEC; ++e) o[e] = v[k + e] * inv_s * invB;
      if (c + VEC > C) {                              // (lanes past C are zeros whatever the row holds)
#pragma unroll
        for (int e = 0; e < VEC; ++e) if (c + e >= C) o[e] = 0.f;
      }
      if (VEC == 4) {
        const __nv_bfloat162 lo = __floats2bfloat162_rn(o[0], o[VEC / 4]), hi = __floats2bfloat162_rn(o[VEC / 2], o[VEC - 1]);
        *reinterpret_cast<uint2*>(d + c) = make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
      } else if (VEC == 2) {
        *reinterpret_cast<__nv_bfloat162*>(d + c) = __floats2bfloat162_rn(o[0], o[VEC - 1]);
      } else {
        d[c] = __float2bfloat16_rn(o[0]);
      }
    }
    if (wide) for (int c = TPR * N + t; c < Cpad; c += TPR) d[c] = __float2bfloat16_rn(c < C ? expf(z[c] - mx) * inv_s * invB : 0.f);
    // A label outside [0, C) comes from caller memory: it must not become an address.  Such a row
    // gets no one-hot term, its loss is NaN (so the minibatch loss is NaN) and the status word, where
    // there is one, records it.
    if (!mine) continue;
    if (unsigned(y) < unsigned(C)) {
      if (t == (y < TPR * N ? y / VEC : y - TPR * N) % TPR) {         // the thread that wrote element y
        const float zy = z[y] - mx;
        d[y] = __float2bfloat16_rn((expf(zy) * inv_s - 1.f) * invB);
        row_loss[row] = -(zy - logf(s));
      }
    } else if (t == 0) {
      row_loss[row] = __int_as_float(0x7fc00000);
      if (status != nullptr) atomicCAS(status, 0, LP_STATUS_BAD_LABEL);
    }
  }
  launch_next();
  if (ticket == nullptr && gridDim.x > 1) return;
  __threadfence();                                    // this block's row losses before its count
  __syncthreads();
  if (threadIdx.x == 0) {
    last = gridDim.x == 1 || atomicInc(ticket, gridDim.x - 1u) == gridDim.x - 1u;     // (wraps to zero: ready for the next launch)
  }
  __syncthreads();
  if (last) {
    __threadfence();
    row_loss_mean<XENT_THREADS>(row_loss, loss_out, B, sh);
  }
}

cudaError_t launch_softmax_xent(const float* zL, int ldz, const int* labels, __nv_bfloat16* delta, int ldd, float* row_loss,
                                unsigned* ticket, float* loss_out, int B, int C, int* status, cudaStream_t stream) {
  const uintptr_t z_at = reinterpret_cast<uintptr_t>(zL), d_at = reinterpret_cast<uintptr_t>(delta);
  const int vec = ldz % 4 == 0 && ldd % 4 == 0 && (z_at & 15) == 0 && (d_at & 7) == 0   ? 4
                  : ldz % 2 == 0 && ldd % 2 == 0 && (z_at & 7) == 0 && (d_at & 3) == 0 ? 2
                                                                                       : 1;
  // Eight threads a row up to 64 classes, a warp up to 1024, a block beyond.  More blocks than are resident at once (four of 64
  // registers a thread) keep an SM's share even; beyond that a block takes several rows.
  const int rows = C <= 64 ? XENT_THREADS / 8 : C <= 1024 ? XENT_THREADS / 32 : 1;
  const int grid = B <= 2 * rows ? 1 : std::min((B + rows - 1) / rows, kSMs * (C <= 1024 ? 8 : 256));
#define LP_XENT(TPR, VEC, N) \
  launch_chained(softmax_xent_kernel<TPR, VEC, N>, grid, XENT_THREADS, 0, stream, 1, zL, ldz, labels, delta, ldd, row_loss, ticket, loss_out, B, C, status)
#define LP_XENT_VEC(TPR, N) (vec == 4 ? LP_XENT(TPR, 4, N) : vec == 2 ? LP_XENT(TPR, 2, N) : LP_XENT(TPR, 1, N))
  const cudaError_t e = C <= 64     ? LP_XENT_VEC(8, 8)
                        : C <= 256  ? LP_XENT_VEC(32, 8)
                        : C <= 1024 ? LP_XENT_VEC(32, 32)
                        : C <= 2048 ? LP_XENT_VEC(256, 8)
                                    : LP_XENT_VEC(256, 32);
#undef LP_XENT_VEC
#undef LP_XENT
  if (e != cudaSuccess || ticket != nullptr || grid == 1) return e;
  return launch_chained(softmax_xent_mean_kernel, 1, XENT_SUMS, 0, stream, 1, static_cast<const float*>(row_loss), loss_out, B);
}

// ---------------------------------------------------------------------------
// Fused update (Eq. 6, optional momentum): m <- mu m + G; W <- W - eta m; ring <- RN(W).
// 8 elements per thread, 128-bit loads and stores throughout.  Blocks past the weight
// range own BIAS_COLS bias columns each: bias gradient = column sums of delta (row order),
// then the same update for the bias.
constexpr int UPD_THREADS = 256;
constexpr int UPD_VEC_PER_THREAD = 2;     // x 8 elements
constexpr int BIAS_COLS = UPD_THREADS / BIAS_LANES;

__global__ void __launch_bounds__(UPD_THREADS) sgd_update_kernel(const UpdateArgs a, int w_blocks) {
  launch_wait();
  if (int(blockIdx.x) < w_blocks) {
    const long long nvec = a.n_elems >> 3;
    const long long base = (long long)blockIdx.x * (UPD_THREADS * UPD_VEC_PER_THREAD) + threadIdx.x;
#pragma unroll
    for (int u = 0; u < UPD_VEC_PER_THREAD; ++u) {
      const long long v = base + (long long)u * UPD_THREADS;
      if (v >= nvec) break;
      const long long e = v << 3;
      const float4 g0 = __ldcs(reinterpret_cast<const float4*>(a.dW + e));
      const float4 g1 = __ldcs(reinterpret_cast<const float4*>(a.dW + e + 4));
      float4 w0 = *reinterpret_cast<const float4*>(a.W + e);
      float4 w1 = *reinterpret_cast<const float4*>(a.W + e + 4);
      float4 m0 = g0, m1 = g1;
      if (a.mW != nullptr) {
        const float4 p0 = *reinterpret_cast<const float4*>(a.mW + e);
        const float4 p1 = *reinterpret_cast<const float4*>(a.mW + e + 4);
        m0.x = a.mu * p0.x + g0.x; m0.y = a.mu * p0.y + g0.y; m0.z = a.mu * p0.z + g0.z; m0.w = a.mu * p0.w + g0.w;
        m1.x = a.mu * p1.x + g1.x; m1.y = a.mu * p1.y + g1.y; m1.z = a.mu * p1.z + g1.z; m1.w = a.mu * p1.w + g1.w;
        *reinterpret_cast<float4*>(a.mW + e) = m0;
        *reinterpret_cast<float4*>(a.mW + e + 4) = m1;
      }
      w0.x -= a.lr * m0.x; w0.y -= a.lr * m0.y; w0.z -= a.lr * m0.z; w0.w -= a.lr * m0.w;
      w1.x -= a.lr * m1.x; w1.y -= a.lr * m1.y; w1.z -= a.lr * m1.z; w1.w -= a.lr * m1.w;
      *reinterpret_cast<float4*>(a.W + e) = w0;
      *reinterpret_cast<float4*>(a.W + e + 4) = w1;
      __nv_bfloat162 q0 = __floats2bfloat162_rn(w0.x, w0.y);
      __nv_bfloat162 q1 = __floats2bfloat162_rn(w0.z, w0.w);
      __nv_bfloat162 q2 = __floats2bfloat162_rn(w1.x, w1.y);
      __nv_bfloat162 q3 = __floats2bfloat162_rn(w1.z, w1.w);
      uint4 o;
      o.x = *reinterpret_cast<uint32_t*>(&q0);
      o.y = *reinterpret_cast<uint32_t*>(&q1);
      o.z = *reinterpret_cast<uint32_t*>(&q2);
      o.w = *reinterpret_cast<uint32_t*>(&q3);
      *reinterpret_cast<uint4*>(a.ring + e) = o;
    }
    return;
  }
  // ---- bias part: this block owns BIAS_COLS columns --------------------------
  __shared__ float part[BIAS_LANES][BIAS_COLS];
  const int cb = (int(blockIdx.x) - w_blocks) * BIAS_COLS;
  const int tx = threadIdx.x % BIAS_COLS, ty = threadIdx.x / BIAS_COLS;
  constexpr int NY = BIAS_LANES;
  const int col = cb + tx;
  float acc = 0.f;
  if (col < a.n_out) {
    for (int r = ty; r < a.rows; r += NY) acc += __bfloat162float(a.delta[(long long)r * a.ldd + col]);
  }
  part[ty][tx] = acc;
  __syncthreads();
  if (ty == 0 && col < a.n_out) {
    float g = 0.f;
#pragma unroll
    for (int i = 0; i < NY; ++i) g += part[i][tx];
    a.db[col] = g;
    float m = g;
    if (a.mb != nullptr) {
      m = a.mu * a.mb[col] + g;
      a.mb[col] = m;
    }
    const float b = a.b[col] - a.lr * m;
    a.b[col] = b;
    a.bring[col] = b;
  }
}

cudaError_t launch_sgd_update(const UpdateArgs& a, cudaStream_t stream) {
  const long long nvec = a.n_elems >> 3;
  const long long per_block = UPD_THREADS * UPD_VEC_PER_THREAD;
  const int w_blocks = int((nvec + per_block - 1) / per_block);
  const int b_blocks = a.delta ? (a.n_out + BIAS_COLS - 1) / BIAS_COLS : 0;
  return launch_chained(sgd_update_kernel, w_blocks + b_blocks, UPD_THREADS, 0, stream, 1, a, w_blocks);
}

}  // namespace lp

namespace lp {
// dst = RN_bf16(src), n a multiple of 8 (used once per layer to seed ring slot 0).
__global__ void round_to_bf16_kernel(const float* __restrict__ src, __nv_bfloat16* __restrict__ dst, long long nvec) {
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < nvec; v += (long long)gridDim.x * blockDim.x) {
    const float4 a = *reinterpret_cast<const float4*>(src + v * 8);
    const float4 b = *reinterpret_cast<const float4*>(src + v * 8 + 4);
    __nv_bfloat162 q0 = __floats2bfloat162_rn(a.x, a.y), q1 = __floats2bfloat162_rn(a.z, a.w);
    __nv_bfloat162 q2 = __floats2bfloat162_rn(b.x, b.y), q3 = __floats2bfloat162_rn(b.z, b.w);
    uint4 o;
    o.x = *reinterpret_cast<uint32_t*>(&q0); o.y = *reinterpret_cast<uint32_t*>(&q1);
    o.z = *reinterpret_cast<uint32_t*>(&q2); o.w = *reinterpret_cast<uint32_t*>(&q3);
    *reinterpret_cast<uint4*>(dst + v * 8) = o;
  }
}
cudaError_t launch_round_to_bf16(const float* src, __nv_bfloat16* dst, long long n_elems, cudaStream_t stream) {
  const long long nvec = n_elems >> 3;
  int blocks = int(std::min<long long>((nvec + 255) / 256, kSMs * 16));
  if (blocks < 1) blocks = 1;
  round_to_bf16_kernel<<<blocks, 256, 0, stream>>>(src, dst, nvec);
  return cudaGetLastError();
}
}  // namespace lp

namespace lp {
// ---------------------------------------------------------------------------
// 2x2 stride-2 max pool, NHWC, 8 channels (16 bytes) per thread.
__global__ void maxpool2_kernel(const __nv_bfloat16* a, __nv_bfloat16* pooled,
                                unsigned char* idx, int B, int H, int W, int C) {
  const int Hp = H / 2, Wp = W / 2, cg = C / 8;
  const long long total = (long long)B * Hp * Wp * cg;
  launch_wait();
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total; t += (long long)gridDim.x * blockDim.x) {
    const int c8 = int(t % cg);
    long long pp = t / cg;
    const int pw = int(pp % Wp);
    const int ph = int((pp / Wp) % Hp);
    const int n = int(pp / ((long long)Wp * Hp));
    float best[8];
    unsigned char bi[8];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const long long src = (((long long)n * H + 2 * ph + (k >> 1)) * W + 2 * pw + (k & 1)) * C + c8 * 8;
      const uint4 v = *reinterpret_cast<const uint4*>(a + src);
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float lo = __uint_as_float(w[j] << 16), hi = __uint_as_float(w[j] & 0xFFFF0000u);
        if (k == 0 || lo > best[2 * j]) { best[2 * j] = lo; bi[2 * j] = (unsigned char)k; }
        if (k == 0 || hi > best[2 * j + 1]) { best[2 * j + 1] = hi; bi[2 * j + 1] = (unsigned char)k; }
      }
    }
    uint4 o;
    uint32_t* ow = reinterpret_cast<uint32_t*>(&o);
#pragma unroll
    for (int j = 0; j < 4; ++j)
      ow[j] = (__float_as_uint(best[2 * j]) >> 16) | (__float_as_uint(best[2 * j + 1]) & 0xFFFF0000u);
    const long long dst = pp * C + c8 * 8;
    *reinterpret_cast<uint4*>(pooled + dst) = o;
    uint2 ib;
    ib.x = bi[0] | (bi[1] << 8) | (bi[2] << 16) | (bi[3] << 24);
    ib.y = bi[4] | (bi[5] << 8) | (bi[6] << 16) | (bi[7] << 24);
    *reinterpret_cast<uint2*>(idx + dst) = ib;
  }
}
cudaError_t launch_maxpool2(const __nv_bfloat16* a, __nv_bfloat16* pooled, unsigned char* idx, int B, int H, int W,
                            int C, cudaStream_t stream) {
  const long long total = (long long)B * (H / 2) * (W / 2) * (C / 8);
  int blocks = int(std::min<long long>((total + 255) / 256, kSMs * 16));
  if (blocks < 1) blocks = 1;
  return launch_chained(maxpool2_kernel, blocks, 256, 0, stream, 1, a, pooled, idx, B, H, W, C);
}

// Bias gradient of a layer with many rows (convolutions, large minibatches): column sums of delta, then Eq. 6 for the
// bias, in one launch.  It is a read of delta at HBM or L2 rate: a thread owns eight columns (one 16-byte load per row) and
// every 32nd row of its block's chunk, four rows in flight; consecutive threads read consecutive
// addresses.  The block adds its 32 row lanes in order and writes one partial sum per column; the last
// block of a 64-column group (a counter that it leaves at zero) adds the chunks in a fixed order and applies the update.
// Device time with cold caches, before (two-byte loads, a second launch for the chunk sums) and now: 802 816 x 128
// 109 + 6 -> 41 us, 3 211 264 x 64 210 + 46 -> 75 us (5.5 TB/s), 2048 x 8192 17 + 4 -> 12 us.
// Narrow matrices: G8 threads of eight columns to a row, as few as cover it, and 256 / G8 row lanes (16 columns read by eight threads
// a row left six of them idle: 1 605 632 x 16 31 -> 18 us, 802 816 x 32 20 -> 17).
template <int G8>
__global__ void __launch_bounds__(256) colsum_bias_kernel(const __nv_bfloat16* x, int rows, int ld, int n_cols, int chunk_rows,
                                                          float* partial, unsigned* counter,
                                                          const BiasUpdate u) {
  constexpr int LANES = 256 / G8;                                  // row lanes
  constexpr int COLS = 8 * G8, PITCH = COLS + 4;
  __shared__ __align__(16) float part[LANES * PITCH > 16 * 68 ? LANES * PITCH : 16 * 68];
  __shared__ bool last;
  const int g = threadIdx.x % G8, lane = threadIdx.x / G8;
  const int col0 = blockIdx.x * 64;
  const int c8 = col0 + g * 8;
  const int r0 = blockIdx.y * chunk_rows, r1 = min(rows, r0 + chunk_rows);
  float acc[8] = {};
  launch_wait();
  if (c8 < ld) {
    const __nv_bfloat16* src = x + c8;
    int r = r0 + lane;
    auto add = [&](const uint4& v) {
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        acc[2 * j] += __uint_as_float(w[j] << 16);
        acc[2 * j + 1] += __uint_as_float(w[j] & 0xFFFF0000u);
      }
    };
    for (; r + 3 * LANES < r1; r += 4 * LANES) {
      uint4 v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = *reinterpret_cast<const uint4*>(src + (long long)(r + k * LANES) * ld);
#pragma unroll
      for (int k = 0; k < 4; ++k) add(v[k]);
    }
    for (; r < r1; r += LANES) add(*reinterpret_cast<const uint4*>(src + (long long)r * ld));
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) part[lane * PITCH + g * 8 + j] = acc[j];
  __syncthreads();
  launch_next();
  constexpr int PER = 256 / COLS;                                  // threads a column, each with its share of the row lanes
  const int tx = threadIdx.x % COLS, ty = threadIdx.x / COLS;
  float s = 0.f;
#pragma unroll
  for (int k = 0; k < LANES / PER; ++k) s += part[(ty * (LANES / PER) + k) * PITCH + tx];
  __syncthreads();
  part[ty * PITCH + tx] = s;
  __syncthreads();
  const int n_chunks = gridDim.y;
  float* mine = partial + (long long)blockIdx.x * n_chunks * 64;   // [chunk][64]
  if (ty == 0) {
    float t = part[tx];
#pragma unroll
    for (int k = 1; k < PER; ++k) t += part[k * PITCH + tx];
    __stcg(mine + blockIdx.y * 64 + tx, t);
    __threadfence();
  }
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(counter + blockIdx.x, 1u) == unsigned(n_chunks) - 1u;
  __syncthreads();
  if (!last) return;
  if (threadIdx.x == 0) counter[blockIdx.x] = 0u;                  // ready for the next launch
  __threadfence();
  const int q = (threadIdx.x & 15) * 4, l16 = threadIdx.x >> 4;    // four columns, every 16th chunk
  float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
  for (int ch = l16; ch < n_chunks; ch += 16) {
    const float4 v = __ldcg(reinterpret_cast<const float4*>(mine + ch * 64 + q));
    t.x += v.x; t.y += v.y; t.z += v.z; t.w += v.w;
  }
  __syncthreads();
  *reinterpret_cast<float4*>(&part[l16 * 68 + q]) = t;
  __syncthreads();
  const int col = col0 + threadIdx.x;
  if (threadIdx.x < 64 && col < n_cols) {
    float grad = 0.f;
#pragma unroll
    for (int k = 0; k < 16; ++k) grad += part[k * 68 + threadIdx.x];
    u.db[col] = grad;
    float m = grad;
    if (u.mb != nullptr) {
      m = u.mu * u.mb[col] + grad;
      u.mb[col] = m;
    }
    const float b = u.b[col] - u.lr * m;
    u.b[col] = b;
    u.bring[col] = b;
  }
}
cudaError_t launch_colsum_bias(const __nv_bfloat16* x, int rows, int ld, int n_cols, float* partial, unsigned* counter,
                               const BiasUpdate& u, cudaStream_t stream) {
  const int chunk = colsum_chunk_rows(rows, n_cols);
  dim3 grid((n_cols + 63) / 64, (rows + chunk - 1) / chunk);
  auto* kernel = ld <= 8 ? colsum_bias_kernel<1> : ld <= 16 ? colsum_bias_kernel<2> : ld <= 32 ? colsum_bias_kernel<4> : colsum_bias_kernel<8>;
  return launch_chained(kernel, grid, 256, 0, stream, 1, x, rows, ld, n_cols, chunk, partial, counter, u);
}
}  // namespace lp

// ---------------------------------------------------------------------------
// lp_softmax_xent_static: the loss kernel for callers that cannot supply scratch memory.
// The per-row losses live in this fixed device array instead of a workspace.  Host code must not pass `g_xent_scratch` itself to a kernel: in host
// code that name is only a handle for the runtime.  The device address is looked up once
// per device with cudaGetSymbolAddress and that pointer is what the kernel receives.
struct XentScratch {
  float row_loss[LP_XENT_STATIC_MAX_BATCH];
};
static __device__ __align__(256) unsigned char g_xent_scratch[sizeof(XentScratch)];

namespace {
constexpr int kMaxDevices = 64;
// device address of the array, per device; written once per device under the mutex, read with acquire
std::atomic<XentScratch*> g_xent_scratch_addr[kMaxDevices];
std::mutex g_xent_setup_mutex;
int xent_fail(int code, const std::string& why) {
  lp::set_global_error("lp_softmax_xent_static: " + why);     // readable through lp_last_error(NULL)
  return code;
}
}  // namespace

extern "C" int lp_softmax_xent_static(const float* logits_dev, int ld_logits, const int* labels_dev,
                                      void* delta_dev, int ld_delta, float* loss_dev, int batch, int classes,
                                      void* stream) {
  if (!logits_dev || !labels_dev || !delta_dev || !loss_dev) return xent_fail(LP_ERR_INVALID_ARG, "null pointer");
  if (batch < 1 || classes < 1) return xent_fail(LP_ERR_INVALID_ARG, "batch and classes must be positive");
  if (batch > LP_XENT_STATIC_MAX_BATCH)     // the fixed scratch holds no more rows
    return xent_fail(LP_ERR_INVALID_ARG, "batch exceeds LP_XENT_STATIC_MAX_BATCH (" + std::to_string(LP_XENT_STATIC_MAX_BATCH) + " rows of built-in scratch)");
  if (ld_logits < classes || ld_delta < ((classes + 7) & ~7))
    return xent_fail(LP_ERR_INVALID_ARG, "row pitch smaller than the (padded) number of classes");
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return xent_fail(LP_ERR_CUDA, "no current CUDA device");
  XentScratch* s = g_xent_scratch_addr[dev].load(std::memory_order_acquire);
  if (s == nullptr) {
    // set-up, once per device, with that device current: ask the runtime where the array lives
    std::lock_guard<std::mutex> lock(g_xent_setup_mutex);
    s = g_xent_scratch_addr[dev].load(std::memory_order_relaxed);
    if (s == nullptr) {
      void* p = nullptr;
      cudaError_t e = cudaGetSymbolAddress(&p, g_xent_scratch);
      if (e != cudaSuccess || p == nullptr) return xent_fail(LP_ERR_CUDA, std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
      s = static_cast<XentScratch*>(p);
      g_xent_scratch_addr[dev].store(s, std::memory_order_release);
    }
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // No counter here: two calls that overlapped could leave anything in it, and clearing it is a launch before the kernel that
  // nothing overlaps with; the mean is a launch behind it, which is in place when the rows are done.
  const cudaError_t e = lp::launch_softmax_xent(logits_dev, ld_logits, labels_dev, static_cast<__nv_bfloat16*>(delta_dev), ld_delta, s->row_loss,
                              nullptr, loss_dev, batch, classes, nullptr, st);
  if (e != cudaSuccess) return xent_fail(LP_ERR_CUDA, std::string("kernel launch: ") + cudaGetErrorString(e));
  return LP_OK;
}
