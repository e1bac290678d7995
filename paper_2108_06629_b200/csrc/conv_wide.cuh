// 3x3 convolution contractions (stride 1) with more than 64 channels on a side, on images tiled by 8 x 16 pixels: forward
// (Eqs. 1-2) and delta (Eqs. 3-4) as an implicit GEMM whose activation operand is fetched once per 64 channels.
//
// The general kernel loads a 128-pixel box and a weight box per (tap, 64-channel chunk): 32 KiB per 256 tensor cycles of a
// 128 x 128 tile, more than an SM gets from L2 (the loads ran at 84 B/clk, the tensor pipe at two thirds).  Here the
// 10 x 18 halo box of a chunk lands in shared memory once and the nine taps are views of it (see conv_halo.cuh), and
// a CTA works on TWO 8 x 16 pixel tiles at a time, so that each 64 x BN weight tap feeds two accumulators: 16 KiB of
// weights and 5 KiB of pixels per 512 cycles.  Two accumulators x two buffers x 128 columns are all of tensor memory;
// with 223 KiB of shared memory no other allocating kernel fits beside a CTA.
//   warp 0     producer: per chunk two halo boxes, then nine weight taps (rings of 2 and 6 stages)
//   warp 1     MMA issuer: per tap four k-slices into either accumulator
//   warps 2-9  epilogue, two warps per tensor-memory quarter, under the next item's main loop
// Persistent CTAs walk the items (pair of pixel tiles, column tile), column tiles fastest: neighbours share pixels in L2.
// 128 -> 128 channels at 112 x 112, batch 64: forward with its pool 235 + 44 -> 206 us, delta 252 -> 237 (the tensor pipe now waits
// for shared memory: 128 columns need all of its 128 B/clk); 4 steps of VGG-16 27.8 -> 27.4 ms.  Not where it is not ahead
// (lp_api.cu): one 64-channel chunk (64 -> 128 forward 175 / 181 us), 64 columns (128 -> 64 delta 267 / 282 before the
// un-pooling epilogue lost its divisions), 256-column tiles of the general kernel (1.3 PFLOP/s there), few items to a CTA.
#pragma once
#include "conv_halo.cuh"

namespace lp {

constexpr int WIDE_A_STAGES = 2;
constexpr int WIDE_A_BYTES = 2 * HALO_BYTES;                   // the halo boxes of both pixel tiles, one 64-channel chunk
constexpr int WIDE_B_STAGES = 6;
constexpr int WIDE_BN = 128;                                   // output columns of a tile
constexpr int WIDE_B_BYTES = WIDE_BN * GEMM_BK * 2;            // one weight tap of a chunk
constexpr int WIDE_THREADS = 320;
constexpr int WIDE_B_OFF = WIDE_A_STAGES * WIDE_A_BYTES;       // 92 160 = 90 KiB
static_assert(WIDE_B_OFF % 1024 == 0, "the weight ring stays 1 KiB aligned");
constexpr int WIDE_SMEM_BYTES = WIDE_B_OFF + WIDE_B_STAGES * WIDE_B_BYTES + 2 * EPI_TILE_BYTES + 256 + 1024;   // 223 KiB: alone on its SM (it holds all of tensor memory)

template <bool B_MN, int MODE>
__global__ void __launch_bounds__(WIDE_THREADS, 1)
conv_wide_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const GemmArgs p,
                 const int tiles_total, const int tiles_n) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  constexpr int BN = WIDE_BN, B_BYTES = WIDE_B_BYTES;
  uint8_t* sB = smem + WIDE_B_OFF;
  float* epi_tile = reinterpret_cast<float*>(sB + WIDE_B_STAGES * B_BYTES);
  uint64_t* bars = reinterpret_cast<uint64_t*>(reinterpret_cast<uint8_t*>(epi_tile) + 2 * EPI_TILE_BYTES);
  uint64_t* afull = bars;
  uint64_t* aempty = afull + WIDE_A_STAGES;
  uint64_t* bfull = aempty + WIDE_A_STAGES;
  uint64_t* bempty = bfull + WIDE_B_STAGES;
  uint64_t* accf = bempty + WIDE_B_STAGES;          // [2]
  uint64_t* acce = accf + 2;                        // [2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acce + 2);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    tma_prefetch_desc(&tmA);
    tma_prefetch_desc(&tmB);
    for (int s = 0; s < WIDE_A_STAGES; ++s) { mbar_init(&afull[s], 1); mbar_init(&aempty[s], 1); }
    for (int s = 0; s < WIDE_B_STAGES; ++s) { mbar_init(&bfull[s], 1); mbar_init(&bempty[s], 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(&accf[b], 1); mbar_init(&acce[b], 8); }
    fence_barrier_init();
  }
  if (warp == 1) {
    if (lane == 0) tmem_note_enter(TK_HALO);
    tmem_alloc(tmem_slot, 512);
    if (lane == 0) tmem_note_got(TK_HALO, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  launch_wait();
  const int items = ((tiles_total + 1) / 2) * tiles_n;
  const int chunks = p.g.chunks_per_tap;
  const int per_image = p.g.tiles_w * p.g.tiles_h;
  // origin of pixel tile t
  auto pixel_tile = [&](int t, TileMap& tm) {
    const int img = t / per_image, r = t - img * per_image, th = r / p.g.tiles_w;
    tm.pn0 = img;
    tm.ph0 = th * 16;
    tm.pw0 = (r - th * p.g.tiles_w) * 8;
  };

  if (warp == 0) {
    if (lane == 0) {
      bool ok = true;
      int ia = 0, ib = 0;                                   // fills issued
      uint32_t as = 0, aph = 0, bs = 0, bph = 0;
      const uint32_t sA0 = smem_u32(smem), sB0 = smem_u32(sB);
      const uint32_t afull0 = smem_u32(afull), aempty0 = smem_u32(aempty), bfull0 = smem_u32(bfull), bempty0 = smem_u32(bempty);
      int it = blockIdx.x;
      for (; it < items && ok; it += gridDim.x) {
        const int tp = it / tiles_n, n0 = p.n_begin + (it - tp * tiles_n) * BN;
        TileMap t0, t1;
        pixel_tile(2 * tp, t0);
        pixel_tile(min(2 * tp + 1, tiles_total - 1), t1);   // (an odd last tile is computed twice, stored once)
        for (int c = 0; c < chunks && ok; ++c) {
          ok = mbar_wait_addr(aempty0 + 8u * as, aph ^ 1u, p.wait_limit);
          if (!ok) break;
          mbar_arrive_expect_tx_addr(afull0 + 8u * as, uint32_t(WIDE_A_BYTES));
          const uint32_t sa = sA0 + as * uint32_t(WIDE_A_BYTES);
          tma_load_4d_addr(sa, &tmA, afull0 + 8u * as, c * 64, t0.pw0 - 1, t0.ph0 - 1, t0.pn0);
          tma_load_4d_addr(sa + HALO_BYTES, &tmA, afull0 + 8u * as, c * 64, t1.pw0 - 1, t1.ph0 - 1, t1.pn0);
          ++ia;
          if (++as == uint32_t(WIDE_A_STAGES)) { as = 0; aph ^= 1u; }
          int col = 0;
          for (int tap = 0; tap < 9; ++tap, col += p.g.tap_pitch) {
            ok = mbar_wait_addr(bempty0 + 8u * bs, bph ^ 1u, p.wait_limit);
            if (!ok) break;
            const uint32_t fb = bfull0 + 8u * bs, sb = sB0 + bs * uint32_t(B_BYTES);
            mbar_arrive_expect_tx_addr(fb, uint32_t(B_BYTES));
            if (B_MN) {        // delta: B[k = (tap, co)][n = ci]
#pragma unroll
              for (int j = 0; j < BN / 64; ++j) tma_load_2d_addr(sb + j * 8192, &tmB, fb, col + n0 + j * 64, c * 64);
            } else {           // forward: B[n = co][k = (tap, ci)]
              tma_load_2d_addr(sb, &tmB, fb, col + c * 64, n0);
            }
            ++ib;
            if (++bs == uint32_t(WIDE_B_STAGES)) { bs = 0; bph ^= 1u; }
          }
        }
      }
      if (!ok) {
        report_expired(p.status, WAIT_WIDE_PRODUCER, it - int(gridDim.x), ib);
        // let copies already in flight land before the CTA's shared memory is released
        for (int i = max(0, ia - WIDE_A_STAGES); i < ia; ++i) mbar_wait(&afull[i % WIDE_A_STAGES], uint32_t(i / WIDE_A_STAGES) & 1u, p.wait_limit);
        for (int i = max(0, ib - WIDE_B_STAGES); i < ib; ++i) mbar_wait(&bfull[i % WIDE_B_STAGES], uint32_t(i / WIDE_B_STAGES) & 1u, p.wait_limit);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t idesc = make_idesc_bf16(GEMM_BM, BN, false, B_MN);
      constexpr uint32_t stepB = (B_MN ? 2048 : 32) >> 4;
      const uint64_t dA = make_smem_desc(smem_u32(smem), 16, HALO_W * 128);
      const uint64_t dB = B_MN ? make_smem_desc(smem_u32(sB), 8192, 1024) : make_smem_desc(smem_u32(sB), 16, 1024);
      const uint32_t dA_hi = uint32_t(dA >> 32), dB_hi = uint32_t(dB >> 32);
      const uint32_t afull0 = smem_u32(afull), aempty0 = smem_u32(aempty), bfull0 = smem_u32(bfull), bempty0 = smem_u32(bempty);
      const uint32_t accf0 = smem_u32(accf), acce0 = smem_u32(acce);
      uint32_t tap_off[9];
#pragma unroll
      for (int tap = 0; tap < 9; ++tap) {
        int r = tap / 3, s = tap % 3;
        if (p.g.flip) { r = 2 - r; s = 2 - s; }
        tap_off[tap] = uint32_t(r * HALO_W + s) * (128u >> 4);
      }
      uint32_t as = 0, aph = 0, bs = 0, bph = 0, n_it = 0;
      bool ok = true;
      int it = blockIdx.x;
      for (; it < items && ok; it += gridDim.x, ++n_it) {
        const uint32_t buf = n_it & 1u;
        ok = mbar_wait_addr(acce0 + 8u * buf, ((n_it >> 1) & 1u) ^ 1u, p.wait_limit);
        if (!ok) break;
        tc_fence_after();
        const uint32_t tacc = tmem_base + buf * 256u;        // accumulators of the two pixel tiles: columns 0 and 128 of the buffer
        uint32_t acc = 0;
        for (int c = 0; c < chunks && ok; ++c) {
          ok = mbar_wait_addr(afull0 + 8u * as, aph, p.wait_limit);
          if (!ok) break;
          const uint32_t a_lo = uint32_t(dA) + as * uint32_t(WIDE_A_BYTES >> 4);
#pragma unroll
          for (int tap = 0; tap < 9; ++tap) {
            if (ok) ok = mbar_wait_addr(bfull0 + 8u * bs, bph, p.wait_limit);
            if (!ok) break;
            tc_fence_after();
            const uint32_t b_lo = uint32_t(dB) + bs * uint32_t(B_BYTES >> 4);
#pragma unroll
            for (int sub = 0; sub < 2; ++sub)
#pragma unroll
              for (int j = 0; j < GEMM_BK / 16; ++j)
                umma_f16_lohi(tacc + sub * 128u, a_lo + uint32_t(sub) * uint32_t(HALO_BYTES >> 4) + tap_off[tap] + uint32_t(j * 2), dA_hi,
                              b_lo + uint32_t(j) * stepB, dB_hi, idesc, acc | uint32_t(j > 0));
            acc = 1;
            umma_commit_addr(bempty0 + 8u * bs);
            if (++bs == uint32_t(WIDE_B_STAGES)) { bs = 0; bph ^= 1u; }
          }
          umma_commit_addr(aempty0 + 8u * as);
          if (++as == uint32_t(WIDE_A_STAGES)) { as = 0; aph ^= 1u; }
        }
        umma_commit_addr(accf0 + 8u * buf);                  // (also releases the epilogue on error)
      }
      if (!ok) report_expired(p.status, WAIT_WIDE_MMA, it - int(gridDim.x), int(bs));
    }
  } else {
    const int q = warp & 3;
    const int half = (warp - 2) >> 2;                        // columns half * BN / 2 .. + BN / 2
    float* tile = epi_tile + (warp - 2) * (32 * EPI_PITCH);
    const int sub_row = lane >> 3, sub_col = (lane & 7) * 4;
    const uint32_t accf0 = smem_u32(accf);
    uint32_t n_it = 0;
    for (int it = blockIdx.x; it < items; it += gridDim.x, ++n_it) {
      const uint32_t buf = n_it & 1u;
      const int tp = it / tiles_n;
      TileMap tm;
      tm.m0 = 0;
      tm.n0 = p.n_begin + (it - tp * tiles_n) * BN;
      tm.nlim = p.N;
      bool ok = mbar_wait_addr(accf0 + 8u * buf, (n_it >> 1) & 1u, p.wait_limit);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) {
        if (lane == 0) report_expired(p.status, WAIT_WIDE_EPILOGUE, it, -1);
        break;
      }
      tc_fence_after();
      const uint32_t tacc = tmem_base + buf * 256u + (uint32_t(q * 32) << 16) + uint32_t(half * (BN / 2));
#pragma unroll 1
      for (int k = 0; k < 2 * (BN / 64); ++k) {              // (pixel tile, 32-column chunk)
        const int sub = k / (BN / 64), c = k % (BN / 64);
        uint32_t r[32];
        __syncwarp();
        tmem_ld_32x32(tacc + uint32_t(sub * 128 + c * 32), r);
        tmem_ld_wait();
        if (k == 2 * (BN / 64) - 1) {                        // last read of this buffer: hand it back to the MMA issuer
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&acce[buf]);
        }
        if (2 * tp + sub >= tiles_total) continue;
#pragma unroll
        for (int g = 0; g < 8; ++g)
          *reinterpret_cast<uint4*>(tile + lane * EPI_PITCH + g * 4) = make_uint4(r[4 * g], r[4 * g + 1], r[4 * g + 2], r[4 * g + 3]);
        __syncwarp();
        pixel_tile(2 * tp + sub, tm);
        epilogue_rows8<MODE>(p, tm, tile, q, sub_row, sub_col, tm.n0 + half * (BN / 2) + c * 32 + sub_col);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
    if (lane == 0) tmem_note_freed(TK_HALO, 512);
  }
}

}  // namespace lp
