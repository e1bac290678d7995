// 3x3 convolution contractions over few channels (at most 64 on both sides): forward
// (Eqs. 1-2) and delta (Eqs. 3-4) as an implicit GEMM whose activation operand is fetched ONCE
// per tile.
//
// The general kernel loads a 128-pixel x 64-channel box per filter tap, i.e. nine shifted copies
// of nearly the same pixels; with only 64 output columns per tile the tensor cores then wait on
// the ~64 B/clk one SM can pull from L2.  Here a tile is 8 x 16 pixels of one image; its
// 10 x 18 halo box (the pixels the nine taps touch) lands in shared memory once (22.5 KiB), and
// the operand of tap (r, s) is a VIEW of it: the matrix descriptor starts r * 10 + s pixel rows
// into the box, eight consecutive pixels of an image row form one 8-row swizzle group and the
// next group is one box row (10 pixels = 1280 bytes) further.  The
// 128-byte swizzle is a function of the absolute shared-memory address for TMA and for the
// tensor core alike, so a view that starts at any 128-byte row of the box needs nothing else
// (checked tap by tap with one-hot weights: exact with the descriptor's base-offset field left
// zero, chunk-permuted when it is set to the start row).  All nine 64 x 64 weight taps stay resident in shared memory (72 KiB) for the whole
// persistent CTA.  Per tile the SM now reads 22.5 KiB instead of 216 KiB; four boxes are in flight.
//
// The same pipeline also runs the forward GEMM of a layer whose whole contraction fits one
// k-block and whose output is at most 64 columns wide (plain geometry: the patch-matrix form of
// a first convolution layer): one weight "tap", tiles of 128 consecutive rows fetched through a
// 2-D map, the output tile stored through a 2-D map.  Such a layer is 25 000 tiles of a single
// k-block each, and what it needs is this kernel's epilogue.
#pragma once
#include "gemm.cuh"

namespace lp {

constexpr int HALO_W = 10, HALO_H = 18;                       // box: pixels per row (pitch) x rows
constexpr int HALO_STAGES = 4;
constexpr int HALO_BYTES = HALO_W * HALO_H * 128;             // 64 bf16 channels per pixel
constexpr int HALO_TAP_BYTES = 64 * 64 * 2;                   // one weight tap: 64 x 64 bf16
constexpr int HALO_OUT_BYTES = GEMM_BM * 128;                 // forward: one output tile, 128 pixels x 64 bf16 channels
constexpr int HALO_THREADS = 320;                             // producer warp, MMA warp, eight epilogue warps
constexpr int HALO_EPI_BYTES = 2 * EPI_TILE_BYTES;            // two output tiles (32 KiB); un-pooling delta: eight transposition tiles (36 KiB)
static_assert(HALO_EPI_BYTES >= 2 * HALO_OUT_BYTES, "the epilogue area holds two output tiles");
constexpr int HALO_SMEM_BYTES = 9 * HALO_TAP_BYTES + HALO_STAGES * HALO_BYTES + HALO_EPI_BYTES + 256 + 1024;
static_assert((HALO_STAGES * HALO_BYTES) % 1024 == 0, "the buffers behind the halo boxes stay 1 KiB aligned");

// SLICES: 16-channel slices of the contraction that exist; the rest of a 64-channel box is zero fill and not multiplied.  A template
// parameter: with a test in front of each MMA the one thread that issues them lost more than it saved.
// TURNS: the epilogue's eight warps are two groups that take the tiles in turn, instead of sharing each tile.  A tile's way from
// accumulator to store is a chain of waits (tensor memory, staging tile free, barriers), and where the MMAs of a tile are
// few -- narrow layers, the patch-matrix form -- that chain is what a tile costs, so two tiles are on it at once.  Times of layers at
// 224 x 224, batch 32, 16 -> 16 channels pooled: forward 134 us with all MMAs, 95 with SLICES, 70 with TURNS; delta 137, 122, 77;
// patch-matrix forward 76, 74, 52.  Wide layers share: 64 -> 64 delta at batch 64 316 us, in turns 333, and the small VGG 1 % slower.
template <bool B_MN, int MODE, int SLICES, bool TURNS>
__global__ void __launch_bounds__(HALO_THREADS, 1)
conv_halo_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                 const __grid_constant__ CUtensorMap tmO, const GemmArgs p, const int tiles_total) {
  constexpr int BN = 64;
  constexpr int HALO_ACC = TURNS ? 4 : 2;               // accumulators: two per group
  constexpr int NGRP = TURNS ? 2 : 1, GW = 8 / NGRP, H = TURNS ? 2 : 1;      // epilogue groups, warps of a group, column halves of a warp
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sB = smem;                                   // [9][64 x 64] weight taps
  uint8_t* sA = smem + 9 * HALO_TAP_BYTES;              // [HALO_STAGES] halo boxes
  uint8_t* sO = sA + HALO_STAGES * HALO_BYTES;                    // forward: [2] output tiles (TMA store sources)
  float* epi_tile = reinterpret_cast<float*>(sO);                 // delta: one transposition tile per epilogue warp (same area)
  uint64_t* bars = reinterpret_cast<uint64_t*>(sO + HALO_EPI_BYTES);
  uint64_t* wfull = bars;          // weights resident
  uint64_t* afull = bars + 1;                       // [HALO_STAGES] halo box landed
  uint64_t* aempty = afull + HALO_STAGES;           // [HALO_STAGES] halo box consumed
  uint64_t* accf = aempty + HALO_STAGES;            // [HALO_ACC] accumulator complete
  uint64_t* acce = accf + HALO_ACC;                 // [HALO_ACC] accumulator drained
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acce + HALO_ACC);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    tma_prefetch_desc(&tmA);
    tma_prefetch_desc(&tmB);
    if (MODE != EPI_DGRAD_UNPOOL) tma_prefetch_desc(&tmO);
    mbar_init(wfull, 1);
    for (int b = 0; b < HALO_STAGES; ++b) {
      mbar_init(&afull[b], 1);
      mbar_init(&aempty[b], 1);
    }
    for (int b = 0; b < HALO_ACC; ++b) {
      mbar_init(&accf[b], 1);
      mbar_init(&acce[b], GW);     // one arrival per warp of the epilogue group
    }
    fence_barrier_init();
  }
  if (warp == 1) {
    if (lane == 0) tmem_note_enter(TK_HALO);
    tmem_alloc(tmem_slot, HALO_ACC * BN);
    if (lane == 0) tmem_note_got(TK_HALO, HALO_ACC * BN);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  launch_wait();
  // CTA b works through the contiguous tile range [t_begin, t_end): neighbouring tiles share halo
  // pixels in L2, and the tile coordinates advance without divisions.
  const bool plain = (p.g.kind == GEOM_PLAIN);          // one tap, 128 consecutive rows per tile
  const int ntaps = plain ? 1 : 9;
  const int tiles_per_image = plain ? 1 : p.g.tiles_w * p.g.tiles_h;
  const int per_cta = (tiles_total + int(gridDim.x) - 1) / int(gridDim.x);
  const int t_begin = min(int(blockIdx.x) * per_cta, tiles_total);
  const int t_end = min(t_begin + per_cta, tiles_total);
  const int tw_begin = plain ? 0 : t_begin % p.g.tiles_w, th_begin = plain ? 0 : (t_begin / p.g.tiles_w) % p.g.tiles_h;
  const int tn_begin = t_begin / tiles_per_image;

  if (warp == 0) {
    if (lane == 0) {
      bool ok = true;
      int issued = 0;
      mbar_arrive_expect_tx(wfull, uint32_t(ntaps) * HALO_TAP_BYTES);
      for (int tap = 0; tap < ntaps; ++tap) tma_load_2d(sB + tap * HALO_TAP_BYTES, &tmB, wfull, tap * p.g.tap_pitch, 0);
      uint32_t st = 0, sph = 0;
      int tw = tw_begin, th = th_begin, n = tn_begin;
      int t = t_begin;
      for (; t < t_end; ++t) {
        ok = mbar_wait(&aempty[st], sph ^ 1u);
        if (!ok) break;
        if (plain) {
          mbar_arrive_expect_tx(&afull[st], GEMM_A_BYTES);
          tma_load_2d(sA + st * HALO_BYTES, &tmA, &afull[st], 0, t * GEMM_BM);
        } else {
          mbar_arrive_expect_tx(&afull[st], HALO_BYTES);
          // the box starts one pixel left of and above the tile; pixels outside the image read zero (= the padding)
          tma_load_4d(sA + st * HALO_BYTES, &tmA, &afull[st], 0, tw * 8 - 1, th * 16 - 1, n);
          if (++tw == p.g.tiles_w) { tw = 0; if (++th == p.g.tiles_h) { th = 0; ++n; } }
        }
        ++issued;
        if (++st == uint32_t(HALO_STAGES)) { st = 0; sph ^= 1u; }
      }
      if (!ok) {
        report_expired(p.status, WAIT_HALO_PRODUCER, t, 0);
        mbar_wait(wfull, 0);
        for (int i = (issued > HALO_STAGES ? issued - HALO_STAGES : 0); i < issued; ++i)
          mbar_wait(&afull[i % HALO_STAGES], uint32_t(i / HALO_STAGES) & 1u);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // (narrow layers: as many accumulator columns as there are channels)
      const uint32_t idesc = TURNS ? idesc_with_cols(make_idesc_bf16(GEMM_BM, BN, false, B_MN), min(BN, (p.N + 15) & ~15))
                                   : make_idesc_bf16(GEMM_BM, BN, false, B_MN);
      constexpr uint32_t stepB = (B_MN ? 2048 : 32) >> 4;
      // One thread issues 36 MMAs per tile, so everything that can be is computed once: the
      // descriptors of box 0 / tap 0, and per tap the start-address offset of its view (the
      // address field counts 16-byte units and never carries out of the low word).
      const uint64_t dA = make_smem_desc(smem_u32(sA), 16, plain ? 1024 : HALO_W * 128);
      const uint64_t dB = B_MN ? make_smem_desc(smem_u32(sB), 8192, 1024) : make_smem_desc(smem_u32(sB), 16, 1024);
      const uint32_t dA_lo0 = uint32_t(dA), dA_hi = uint32_t(dA >> 32), dB_lo0 = uint32_t(dB), dB_hi = uint32_t(dB >> 32);
      uint32_t tap_off[9];
#pragma unroll
      for (int tap = 0; tap < 9; ++tap) {
        int r = tap / 3, s = tap % 3;
        if (p.g.flip) { r = 2 - r; s = 2 - s; }        // delta: the tap's shift is mirrored
        tap_off[tap] = uint32_t(r * HALO_W + s) * (128u >> 4);
      }
      bool ok = mbar_wait(wfull, 0);
      uint32_t it = 0, st = 0, sph = 0;
      int t = t_begin;
      for (; t < t_end && ok; ++t, ++it) {
        const uint32_t buf = it % HALO_ACC;
        ok = mbar_wait(&acce[buf], ((it / HALO_ACC) & 1u) ^ 1u);
        if (!ok) break;
        ok = mbar_wait(&afull[st], sph);
        if (!ok) break;
        tc_fence_after();
        const uint32_t tacc = tmem_base + buf * uint32_t(BN);
        const uint32_t a_lo = dA_lo0 + st * uint32_t(HALO_BYTES >> 4);
        uint32_t acc = 0;
#pragma unroll
        for (int tap = 0; tap < 9; ++tap) {
          if (tap >= ntaps) break;
#pragma unroll
          for (int j = 0; j < SLICES; ++j) {
            umma_f16_lohi(tacc, a_lo + tap_off[tap] + uint32_t(j * 2), dA_hi,
                          dB_lo0 + uint32_t(tap) * uint32_t(HALO_TAP_BYTES >> 4) + uint32_t(j) * stepB, dB_hi, idesc, acc);
            acc = 1;
          }
        }
        umma_commit(&aempty[st]);
        umma_commit(&accf[buf]);
        if (++st == uint32_t(HALO_STAGES)) { st = 0; sph ^= 1u; }
      }
      if (!ok) report_expired(p.status, WAIT_HALO_MMA, t, 0);
    }
  } else {
    // Warp w reads tensor-memory lanes 32 * (w % 4) (the rows of its quarter of the tile), a lane one row: 32 columns of
    // it where all eight warps share a tile, else all of it.  With one warp per scheduler there is nothing to
    // hide an instruction's latency behind, so the epilogue is spread as wide as the tile allows.
    const int q = warp & 3;
    const int grp = (warp - 2) / GW, half0 = TURNS ? 0 : (warp - 2) >> 2;
    float* tile = epi_tile + (warp - 2) * (32 * EPI_PITCH);
    const int sub_row = lane >> 3;
    const int sub_col = (lane & 7) * 4;
    const bool chief = threadIdx.x == 64u + 32u * uint32_t(GW * grp);    // issues its group's stores
    auto group_sync = [&] { asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "n"(32 * GW) : "memory"); };
    uint32_t it = uint32_t(grp);
    bool dead = false;      // a wait ran out: keep the named-barrier count, touch nothing else
    const int halves = TURNS ? min((p.N + 31) / 32, 2) : 1;          // of this warp's column halves, those with output channels
    // the bias of this warp's output channels does not depend on the tile (rows are padded to 8 with zeros)
    float4 bias4[8 * H];
#pragma unroll
    for (int g = 0; g < 8 * H; ++g) {
      const int n = half0 * 32 + 4 * g;
      bias4[g] = (MODE == EPI_FPROP && p.bias != nullptr && n < p.N) ? *reinterpret_cast<const float4*>(p.bias + n)
                                                                     : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    int tw = tw_begin, th = th_begin, tn = tn_begin;
    auto next_tile = [&] { if (!plain && ++tw == p.g.tiles_w) { tw = 0; if (++th == p.g.tiles_h) { th = 0; ++tn; } } };
    if (grp == 1) next_tile();
    // delta: what f' is evaluated on, this lane's pixel and columns, asked for one tile of the group ahead: an accumulator is
    // usually complete when these warps reach it, and the round trip would be theirs alone
    constexpr int kAux = MODE == EPI_DGRAD ? 4 * H : 1;
    uint4 av[kAux], av_next[kAux];
    auto load_aux = [&](int t, uint4 (&v)[kAux]) {
      const int img = t / tiles_per_image, r = t - img * tiles_per_image, rh = r / p.g.tiles_w;
      const int trow = q * 32 + lane;
      const size_t pix = (size_t(img) * p.g.H + rh * 16 + (trow >> 3)) * p.g.W + (r - rh * p.g.tiles_w) * 8 + (trow & 7);
      const __nv_bfloat16* src = p.aux + pix * p.ld_aux + half0 * 32;
#pragma unroll
      for (int u = 0; u < kAux; ++u)
        v[u] = (p.act != ACT_NONE && half0 * 32 + 8 * u < p.ld_aux) ? *reinterpret_cast<const uint4*>(src + 8 * u) : make_uint4(0u, 0u, 0u, 0u);
    };
    if (MODE == EPI_DGRAD && t_begin + grp < t_end) load_aux(t_begin + grp, av_next);
    for (int t = t_begin + grp; t < t_end; t += NGRP, it += NGRP) {
      const uint32_t buf = it % HALO_ACC;
      if constexpr (MODE == EPI_DGRAD) {
#pragma unroll
        for (int u = 0; u < kAux; ++u) av[u] = av_next[u];
        if (t + NGRP < t_end) load_aux(t + NGRP, av_next);
      }
      TileMap tm;
      tm.m0 = t * GEMM_BM;            // (plain geometry)
      tm.n0 = 0;
      tm.nlim = p.N;
      tm.pw0 = tw * 8;
      tm.ph0 = th * 16;
      tm.pn0 = tn;
#pragma unroll
      for (int k = 0; k < NGRP; ++k) next_tile();
      if (!dead) {
        bool ok = mbar_wait(&accf[buf], (it / HALO_ACC) & 1u);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) {
          if (lane == 0) report_expired(p.status, WAIT_HALO_EPILOGUE, t, -1);
          dead = true;
        }
      }
      if (dead && MODE == EPI_DGRAD_UNPOOL) break;      // the other epilogues have barriers of the group
      tc_fence_after();
      const uint32_t tacc = tmem_base + buf * uint32_t(BN) + (uint32_t(q * 32) << 16);
      if constexpr (MODE != EPI_DGRAD_UNPOOL) {
        // A lane keeps its accumulator row (one pixel), adds the bias and applies f (forward) or multiplies by
        // f' (delta), and writes the 64 bf16 channels as one 128-byte swizzled row of a shared-memory tile that a
        // TMA store sends to the NHWC output (8 x 16 pixel box) -- no transposition, no address
        // arithmetic per element, and the global writes are whole lines.  (Delta through transposition
        // tiles and 8-byte accesses: 418 us for 64 channels at 224 x 224, batch 64; this form 314, 428 without the look-ahead.)
        const int trow = q * 32 + lane;
        const uint32_t stage = smem_u32(sO) + (TURNS ? uint32_t(grp) : buf) * uint32_t(HALO_OUT_BYTES);
        const uint32_t so = stage + uint32_t(trow) * 128u;
        const uint32_t swz = uint32_t(trow & 7);
        uint32_t packed[16];
        auto compute = [&](int h) {                     // h: which of this warp's column halves
          uint32_t r[32];
          tmem_ld_32x32(tacc + uint32_t((half0 + h) * 32), r);
          tmem_ld_wait();
          if (h == halves - 1) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acce[buf]);
          }
#pragma unroll
          for (int g = 0; g < 8; ++g) {
            const int n = (half0 + h) * 32 + 4 * g;
            float v[4] = {__uint_as_float(r[4 * g]), __uint_as_float(r[4 * g + 1]), __uint_as_float(r[4 * g + 2]), __uint_as_float(r[4 * g + 3])};
            uint32_t a01 = 0u, a23 = 0u;
            if constexpr (MODE == EPI_FPROP) {
              const float4 b = bias4[h * 8 + g];
              v[0] += b.x; v[1] += b.y; v[2] += b.z; v[3] += b.w;
            } else {
              const uint4 a = av[h * 4 + (g >> 1)];
              a01 = (g & 1) ? a.z : a.x;
              a23 = (g & 1) ? a.w : a.y;
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              if (n + e >= p.N) v[e] = 0.f;
              else if (MODE == EPI_FPROP) { if (p.act == ACT_RELU) v[e] = fmaxf(v[e], 0.f); }
              else if (p.act != ACT_NONE) {
                const float z = (e & 1) ? bf16_hi(e < 2 ? a01 : a23) : bf16_lo(e < 2 ? a01 : a23);
                v[e] = p.act == ACT_RELU ? (z > 0.f ? v[e] : 0.f) : v[e] * gelu_grad(z);
              }
            }
            packed[2 * g] = pack_bf16x2(v[0], v[1]);
            packed[2 * g + 1] = pack_bf16x2(v[2], v[3]);
          }
        };
        auto put = [&](int h) {
#pragma unroll
          for (int u = 0; u < 4; ++u)
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(so + ((uint32_t((half0 + h) * 4 + u) ^ swz) << 4)), "r"(packed[4 * u]),
                         "r"(packed[4 * u + 1]), "r"(packed[4 * u + 2]), "r"(packed[4 * u + 3])
                         : "memory");
        };
        if (!TURNS && !dead) compute(0);
        // the staging tile must have been read by its last store -- the group's last, or that of two tiles ago -- and by the
        // threads that pooled it
        if (chief) {
          if (TURNS) tma_store_wait_read0();
          else       asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
        }
        group_sync();
        if (TURNS && !dead) {
#pragma unroll
          for (int h = 0; h < H; ++h) {
            if (h >= halves) break;
            compute(h);
            put(h);
          }
        }
        if (!TURNS && !dead) put(0);
        if (MODE == EPI_FPROP && p.pool_out_idx != nullptr) {
          // 2x2 max pool of the staged tile: a thread takes eight channels of one of its 32 windows, or of two
          group_sync();
#pragma unroll
          for (int k2 = 0; k2 < H; ++k2) {
            const int e = ((int(threadIdx.x) - 64) & (32 * GW - 1)) + k2 * (32 * GW), pp = e >> 3, cg = e & 7;
            if (dead || cg * 8 >= p.ld_out) continue;
            const int pw = pp & 3, ph = pp >> 2;
            float best[8];
            uint32_t idx[2] = {0u, 0u};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const uint32_t tr = uint32_t((2 * ph + (k >> 1)) * 8 + 2 * pw + (k & 1));
              uint32_t w[4];
              asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3])
                           : "r"(stage + tr * 128u + ((uint32_t(cg) ^ (tr & 7u)) << 4)));
#pragma unroll
              for (int j = 0; j < 4; ++j) pool_step(w[j], k, best + 4 * (j >> 1), idx[j >> 1], 2 * (j & 1));
            }
            const size_t off = (size_t(tm.pn0 * p.pool_Hp + (tm.ph0 >> 1) + ph) * p.pool_Wp + (tm.pw0 >> 1) + pw) * p.ld_out + cg * 8;
            *reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(p.out) + off) =
                make_uint4(pool_pack(best), pool_pack(best + 2), pool_pack(best + 4), pool_pack(best + 6));
            *reinterpret_cast<uint2*>(p.pool_out_idx + off) = make_uint2(idx[0], idx[1]);
          }
          continue;
        }
        fence_proxy_async_smem();
        group_sync();
        if (chief && !dead) {
          if (plain) {
            tma_store_2d_addr(&tmO, stage, 0, tm.m0);
          } else {
            asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.tile.bulk_group [%0, {%2, %3, %4, %5}], [%1];" ::"l"(
                             reinterpret_cast<uint64_t>(&tmO)),
                         "r"(stage), "r"(0), "r"(tm.pw0), "r"(tm.ph0), "r"(tm.pn0)
                         : "memory");
          }
          tma_store_commit();
        }
        continue;
      }
#pragma unroll 1
      for (int h = 0; h < halves; ++h) {
        const int c = half0 + h;
        uint32_t r[32];
        __syncwarp();
        tmem_ld_32x32(tacc + uint32_t(c * 32), r);
        tmem_ld_wait();
        if (h == halves - 1) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&acce[buf]);
        }
#pragma unroll
        for (int g = 0; g < 8; ++g)
          *reinterpret_cast<uint4*>(tile + lane * EPI_PITCH + g * 4) = make_uint4(r[4 * g], r[4 * g + 1], r[4 * g + 2], r[4 * g + 3]);
        __syncwarp();
        epilogue_rows8<MODE>(p, tm, tile, q, sub_row, sub_col, c * 32 + sub_col);
      }
    }
    if (MODE != EPI_DGRAD_UNPOOL && chief) tma_store_wait_read0();   // shared memory must outlive the stores' reads
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, HALO_ACC * BN);
    if (lane == 0) tmem_note_freed(TK_HALO, HALO_ACC * BN);
  }
}

// ---------------------------------------------------------------------------------------------
// G (Eq. 5) of the same layers: G[co][tap][ci] = sum over pixels of delta[px][co] a[px + tap][ci].
//
// The general kernel gives every (tap, 64-pixel k-block) its own pair of TMA loads, so the nine
// taps re-read delta and the activations nine times through L2, and with 64 output channels
// only half of each 128-row MMA is used.  Here the contraction runs over 8 x 16 pixel tiles:
// per tile one delta box (128 pixels x 64 channels, 16 KiB) and one activation halo box
// (22.5 KiB) are fetched, and the TRANSPOSED gradient is accumulated,
//   D[m = (tap pair half, ci)][n = co] += sum_px  A[px][m] B[px][n],
// with A = two shifted views of the halo box side by side (the descriptor's leading-dimension
// stride, the distance between the two 64-wide halves of M, is the distance between the two
// taps: one pixel = 128 bytes, or 1024 bytes from tap (r, 2) to tap (r + 1, 0)) and B = the delta
// box.  Nine taps = four pairs and a single: five accumulators of 64 columns stay in tensor
// memory over ALL tiles of the CTA; at the end each CTA writes its 5 x 128 x 64 partial sums and
// a second small kernel adds the CTAs' partials in CTA order and applies Eq. 6.  A layer with
// 128 output channels takes two such passes (64 channels each).
constexpr int HALOG_STAGES = 5;                                 // 201 KiB: this CTA takes all 512 tensor-memory columns, so no other kernel that allocates any may fit beside it
constexpr int HALOG_D_OFF = 24576;                              // delta box behind the halo box (1 KiB aligned)
constexpr int HALOG_STAGE_BYTES = HALOG_D_OFF + GEMM_A_BYTES;   // 40 KiB
constexpr int HALOG_SMEM_BYTES = HALOG_STAGES * HALOG_STAGE_BYTES + 256 + 1024;
constexpr int HALOG_GROUPS = 5;
constexpr int HALOG_PART_FLOATS = HALOG_GROUPS * GEMM_BM * 64;  // partial sums of one CTA

template <int kInstance = 0>   // (a template only so that the header may be included by several translation units)
__global__ void __launch_bounds__(GEMM_THREADS, 1)
conv_halo_g_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmD, const ConvGeom g,
                   const int tiles_total, const int co0, float* partial, int* status) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + HALOG_STAGES * HALOG_STAGE_BYTES);
  uint64_t* full = bars;
  uint64_t* empty = bars + HALOG_STAGES;
  uint64_t* accf = empty + HALOG_STAGES;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(accf + 1);
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    tma_prefetch_desc(&tmX);
    tma_prefetch_desc(&tmD);
    for (int b = 0; b < HALOG_STAGES; ++b) {
      mbar_init(&full[b], 1);
      mbar_init(&empty[b], 1);
    }
    mbar_init(accf, 1);
    fence_barrier_init();
  }
  if (warp == 1) {
    if (lane == 0) tmem_note_enter(TK_HALO_G);
    tmem_alloc(tmem_slot, 512);
    if (lane == 0) tmem_note_got(TK_HALO_G, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  launch_wait();
  const int per_cta = (tiles_total + int(gridDim.x) - 1) / int(gridDim.x);
  const int t_begin = min(int(blockIdx.x) * per_cta, tiles_total);
  const int t_end = min(t_begin + per_cta, tiles_total);

  if (warp == 0) {
    if (lane == 0) {
      bool ok = true;
      int issued = 0;
      uint32_t st = 0, sph = 0;
      int tw = t_begin % g.tiles_w, th = (t_begin / g.tiles_w) % g.tiles_h, n = t_begin / (g.tiles_w * g.tiles_h);
      int t = t_begin;
      for (; t < t_end; ++t) {
        ok = mbar_wait(&empty[st], sph ^ 1u);
        if (!ok) break;
        uint8_t* base = smem + st * HALOG_STAGE_BYTES;
        mbar_arrive_expect_tx(&full[st], HALO_BYTES + GEMM_A_BYTES);
        tma_load_4d(base, &tmX, &full[st], 0, tw * 8 - 1, th * 16 - 1, n);
        tma_load_4d(base + HALOG_D_OFF, &tmD, &full[st], co0, tw * 8, th * 16, n);   // 64 output channels from co0
        ++issued;
        if (++st == uint32_t(HALOG_STAGES)) { st = 0; sph ^= 1u; }
        if (++tw == g.tiles_w) { tw = 0; if (++th == g.tiles_h) { th = 0; ++n; } }
      }
      if (!ok) {
        report_expired(status, WAIT_HALO_G_PRODUCER, t, 0);
        for (int i = (issued > HALOG_STAGES ? issued - HALOG_STAGES : 0); i < issued; ++i)
          mbar_wait(&full[i % HALOG_STAGES], uint32_t(i / HALOG_STAGES) & 1u);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t idesc = make_idesc_bf16(GEMM_BM, 64, true, true);      // (fewer columns for narrow layers gain nothing: the MMAs wait for A)
      // tap groups: first tap of the group as a halo row offset, and the distance to its partner
      const uint32_t first_row[HALOG_GROUPS] = {0u, 2u, uint32_t(HALO_W + 1), uint32_t(2 * HALO_W), uint32_t(2 * HALO_W + 2)};
      const uint32_t lbo[HALOG_GROUPS] = {128u, uint32_t((HALO_W - 2) * 128), 128u, 128u, 0u};
      uint32_t dA_lo[HALOG_GROUPS], dA_hi[HALOG_GROUPS];
#pragma unroll
      for (int q = 0; q < HALOG_GROUPS; ++q) {
        const uint64_t d = make_smem_desc(smem_u32(smem) + first_row[q] * 128u, lbo[q], HALO_W * 128);
        dA_lo[q] = uint32_t(d);
        dA_hi[q] = uint32_t(d >> 32);
      }
      const uint64_t dB = make_smem_desc(smem_u32(smem) + HALOG_D_OFF, 8192, 1024);
      const uint32_t dB_lo0 = uint32_t(dB), dB_hi = uint32_t(dB >> 32);
      bool ok = true;
      uint32_t st = 0, sph = 0, acc = 0;
      int t = t_begin;
      for (; t < t_end; ++t) {
        ok = mbar_wait(&full[st], sph);
        if (!ok) break;
        tc_fence_after();
        const uint32_t soff = st * uint32_t(HALOG_STAGE_BYTES >> 4);
#pragma unroll
        for (int k = 0; k < 8; ++k) {            // 16 pixels per MMA: two image rows of the tile
#pragma unroll
          for (int q = 0; q < HALOG_GROUPS; ++q)
            umma_f16_lohi(tmem_base + uint32_t(q * 64), dA_lo[q] + soff + uint32_t(k) * uint32_t((2 * HALO_W * 128) >> 4), dA_hi[q],
                          dB_lo0 + soff + uint32_t(k) * (2048u >> 4), dB_hi, idesc, acc);
          acc = 1;
        }
        umma_commit(&empty[st]);
        if (++st == uint32_t(HALOG_STAGES)) { st = 0; sph ^= 1u; }
      }
      if (!ok) report_expired(status, WAIT_HALO_G_MMA, t, 0);
      umma_commit(accf);
    }
  } else {
    const int q = warp & 3;
    bool ok = mbar_wait(accf, 0);
    ok = __all_sync(0xffffffffu, ok);
    if (!ok && lane == 0) report_expired(status, WAIT_HALO_G_EPILOGUE, t_begin, -1);
    tc_fence_after();
    float* dst = partial + size_t(blockIdx.x) * HALOG_PART_FLOATS;
    const bool any = t_end > t_begin;          // a CTA without tiles contributes zeros
    for (int grp = 0; grp < HALOG_GROUPS; ++grp) {
#pragma unroll 1
      for (int c = 0; c < 2; ++c) {
        uint32_t r[32];
        if (ok && any) {
          tmem_ld_32x32(tmem_base + (uint32_t(q * 32) << 16) + uint32_t(grp * 64 + c * 32), r);
          tmem_ld_wait();
        } else {
#pragma unroll
          for (int j = 0; j < 32; ++j) r[j] = 0u;
        }
        float4* o = reinterpret_cast<float4*>(dst + (size_t(grp) * GEMM_BM + q * 32 + lane) * 64 + c * 32);
#pragma unroll
        for (int j = 0; j < 8; ++j)
          o[j] = make_float4(__uint_as_float(r[4 * j]), __uint_as_float(r[4 * j + 1]), __uint_as_float(r[4 * j + 2]), __uint_as_float(r[4 * j + 3]));
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
    if (lane == 0) tmem_note_freed(TK_HALO_G, 512);
  }
}

// Adds the CTAs' partial sums and applies Eq. 6 (or only stores G when W is null).  A block owns 32 elements of the
// transposed accumulators, n (= output channel) fastest, so the partial sums are read coalesced; its eight warps
// add every eighth CTA's in CTA order, and the warp sums follow in order (one thread per element went through all
// 148 partials alone: 18 us).  The 64 x 9 x 64 weight elements themselves are scattered.
struct HaloGUpdate {
  const float* partial;
  int n_ctas;
  int co0;                        // first output channel of this pass (layers with more than 64 take several)
  int n_out, n_in, ld_w;          // weight matrix [n_out][9 * tap_pitch], pitch ld_w
  int tap_pitch;
  float* G;                       // may be null
  float* W;                       // null: store G only
  float* mW;                      // may be null
  __nv_bfloat16* ring;
  float lr, mu;
};
template <int kInstance = 0>
__global__ void __launch_bounds__(256) conv_halo_g_update_kernel(const HaloGUpdate a) {
  __shared__ float sums[8][32];
  const int lane = threadIdx.x & 31, wrp = threadIdx.x >> 5;
  const int e = blockIdx.x * 32 + lane;              // (the partial tile is a whole number of blocks)
  const float* src = a.partial + e;
  float g = 0.f;
  launch_wait();
#pragma unroll 8
  for (int c = wrp; c < a.n_ctas; c += 8) g += __ldcg(src + size_t(c) * HALOG_PART_FLOATS);
  sums[wrp][lane] = g;
  __syncthreads();
  if (wrp != 0) return;
#pragma unroll
  for (int k = 1; k < 8; ++k) g += sums[k][lane];
  const int co = a.co0 + (e & 63), m = (e >> 6) & 127, grp = e >> 13;
  const int half = m >> 6, ci = m & 63;
  const int tap = (grp < 4) ? 2 * grp + half : (half == 0 ? 8 : -1);
  if (tap < 0 || ci >= a.n_in || co >= a.n_out) return;
  const size_t off = size_t(co) * a.ld_w + size_t(tap) * a.tap_pitch + ci;
  if (a.G != nullptr) a.G[off] = g;
  if (a.W == nullptr) return;
  float mm = g;
  if (a.mW != nullptr) {
    mm = a.mu * a.mW[off] + g;
    a.mW[off] = mm;
  }
  const float w = a.W[off] - a.lr * mm;
  a.W[off] = w;
  a.ring[off] = __float2bfloat16_rn(w);
}

}  // namespace lp
