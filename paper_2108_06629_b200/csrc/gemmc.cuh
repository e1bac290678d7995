// Contraction split over the CTAs of a cluster, for outputs of few tiles (small minibatches, narrow layers).
//
// Such a launch is bound by latency: a 256 x 4096 output is 64 tiles of 128 x 128, each a serial chain of 64
// k-blocks, on 148 SMs; a 32 x 256 one is two tiles.  Here the C CTAs of a cluster share one 128 x BN tile: CTA r contracts the
// r-th contiguous range of k-blocks into its own tensor memory, writes the fp32 partial tile to its shared memory (over
// the operand ring, which has been read by then), and after one cluster barrier every CTA adds the C partial
// tiles of ITS share of the elements through distributed shared memory, in rank order -- a fixed order, so results
// do not depend on timing -- and runs the epilogue on them.  The chain of k-blocks and the epilogue both
// shrink by C, nothing goes through global memory (the split-K form of gemm.cuh writes and re-reads its partial tiles there and
// leaves the sum and the epilogue to a second launch).  A cluster of one is the same without the sum: 64-column tiles and all
// six warps in the epilogue (32 x 256 x 10 5.1 -> 3.1 us, 1000 x 900 x 1000 13.5 -> 9.3 against the 128-column form of gemm.cuh).
//
// SEGS: consecutive parts of a CTA's k-blocks with an accumulator of their own, which the epilogue adds in order.  The tensor
// core truncates the running sum once per 16 terms, so the error grows with the length of a chain; SEGS keeps the chains as short as
// a division over more CTAs has them where fewer CTAs are the faster ones.
#pragma once
#include "gemm2.cuh"

namespace lp {

constexpr int gemmc_part_pitch(int bn) { return bn + 4; }      // floats; 16-byte accesses of eight consecutive rows touch all banks
constexpr int gemmc_stages(int bn) { return bn <= 64 ? 4 : 3; }   // 96 KiB: two CTAs per SM
constexpr int gemmc_smem_bytes(int bn) { return gemmc_stages(bn) * (GEMM_A_BYTES + bn * GEMM_BK * 2) + 256 + 1024; }

__device__ __forceinline__ float4 ld_cluster_f4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}

// This CTA's share of the tile: groups of four consecutive columns, dealt to the cluster's threads in order.
template <int BN, int MODE, int C>
__device__ __forceinline__ void gemmc_reduce_store(const GemmArgs& p, const TileMap& tm, uint32_t part, uint32_t rank) {
  constexpr int U = 4;                                  // groups in flight per thread
  const int rows = min(GEMM_BM, p.M - tm.m0);
  const int total = rows * (BN / 4);
  const int step = C * GEMM_THREADS;
  const int n_pad8 = (tm.nlim + 7) & ~7;
  for (int g0 = int(rank) * GEMM_THREADS + int(threadIdx.x); g0 < total; g0 += U * step) {
    float4 acc[U];
    uint2 av[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int g = g0 + u * step;
      const int row = tm.m0 + g / (BN / 4), n = tm.n0 + (g % (BN / 4)) * 4;
      av[u] = make_uint2(0u, 0u);
      if (MODE == EPI_DGRAD && p.act != ACT_NONE && g < total && n < n_pad8)
        av[u] = *reinterpret_cast<const uint2*>(p.aux + size_t(row) * p.ld_aux + n);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int g = min(g0 + u * step, total - 1);
      const uint32_t a = part + uint32_t((g / (BN / 4)) * gemmc_part_pitch(BN) + (g % (BN / 4)) * 4) * 4u;
      float4 t[C];
#pragma unroll
      for (int r = 0; r < C; ++r) t[r] = ld_cluster_f4(map_to_cta(a, uint32_t(r)));
      acc[u] = t[0];
#pragma unroll
      for (int r = 1; r < C; ++r) {
        acc[u].x += t[r].x; acc[u].y += t[r].y; acc[u].z += t[r].z; acc[u].w += t[r].w;
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int g = g0 + u * step;
      if (g >= total) continue;
      const int row = tm.m0 + g / (BN / 4), n = tm.n0 + (g % (BN / 4)) * 4;
      if constexpr (MODE == EPI_DGRAD) {
        if (n >= n_pad8) continue;
        const float v[4] = {n + 0 < tm.nlim ? acc[u].x : 0.f, n + 1 < tm.nlim ? acc[u].y : 0.f, n + 2 < tm.nlim ? acc[u].z : 0.f,
                            n + 3 < tm.nlim ? acc[u].w : 0.f};
        dgrad_store4(p, row, n, v, av[u]);
      } else {
        epilogue_store4<MODE>(p, row, n, tm.nlim, acc[u]);
      }
    }
  }
}

// ONE: a cluster of one (a kernel of its own: one more case in the switch at the end slowed the others, the ragged GELU MLP 627 -> 637 us)
template <int BN, bool A_MN, bool B_MN, int MODE, bool ONE, int SEGS>
__global__ void __launch_bounds__(GEMM_THREADS, 2)
gemmc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const GemmArgs p, const int tiles_m) {
  static_assert(MODE != EPI_WGRAD_UPDATE, "the update has tiles enough");
  using SM = GemmSmem<BN>;
  constexpr int S = gemmc_stages(BN);
  static_assert(S * SM::STAGE_BYTES >= GEMM_BM * gemmc_part_pitch(BN) * 4, "the partial tile reuses the operand ring");
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full_bar = reinterpret_cast<uint64_t*>(smem + size_t(S) * SM::STAGE_BYTES);
  uint64_t* empty_bar = full_bar + S;
  uint64_t* acc_bar = empty_bar + S;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_bar + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int C = ONE ? 1 : p.cluster;
  TileMap tm;
  tm.m0 = (int(blockIdx.y) % tiles_m) * GEMM_BM;
  tm.n0 = p.n_begin + (int(blockIdx.y) / tiles_m) * BN;
  tm.nlim = p.N;
  tm.pn0 = tm.ph0 = tm.pw0 = 0;
  const int kb_total = (p.K + GEMM_BK - 1) / GEMM_BK;
  const int kb_each = kb_total / C, kb_more = kb_total % C;       // the first kb_more ranks take one more
  const int kb0 = int(rank) * kb_each + min(int(rank), kb_more);
  const int num_kb = kb_each + (int(rank) < kb_more ? 1 : 0);     // (at least one a part: gemm_pick_cluster)

  if (threadIdx.x == 0) {
    tma_prefetch_desc(&tmA);
    tma_prefetch_desc(&tmB);
    for (int s = 0; s < S; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], 1);
    }
    mbar_init(acc_bar, 1);
    fence_barrier_init();
  }
  if (warp == 1) {
    if (lane == 0) tmem_note_enter(TK_GEMM);
    tmem_alloc(tmem_slot, BN * SEGS);
    if (lane == 0) tmem_note_got(TK_GEMM, BN * SEGS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  launch_wait();
  const uint32_t full0 = smem_u32(full_bar), empty0 = smem_u32(empty_bar);

  if (warp == 0) {
    if (lane == 0) {
      bool ok = true;
      int issued = 0;
      const uint32_t smem0 = smem_u32(smem);
      uint32_t s = 0, ph = 0;
      int k0 = kb0 * GEMM_BK, kb = 0;
      for (; kb < num_kb; ++kb, k0 += GEMM_BK) {
        ok = mbar_wait_addr(empty0 + 8u * s, ph ^ 1u, p.wait_limit);
        if (!ok) break;
        const uint32_t sa = smem0 + s * uint32_t(SM::STAGE_BYTES), sb = sa + GEMM_A_BYTES, fb = full0 + 8u * s;
        mbar_arrive_expect_tx_addr(fb, SM::STAGE_BYTES);
        if (B_MN) {
#pragma unroll
          for (int c = 0; c < BN / 64; ++c) tma_load_2d_addr(sb + c * 8192, &tmB, fb, tm.n0 + c * 64, k0);
        } else {
          tma_load_2d_addr(sb, &tmB, fb, k0, tm.n0);
        }
        if (A_MN) {
#pragma unroll
          for (int c = 0; c < GEMM_BM / 64; ++c) tma_load_2d_addr(sa + c * 8192, &tmA, fb, tm.m0 + c * 64, k0);
        } else {
          tma_load_2d_addr(sa, &tmA, fb, k0, tm.m0);
        }
        ++issued;
        if (++s == uint32_t(S)) { s = 0; ph ^= 1u; }
      }
      launch_next();
      if (!ok) {
        report_expired(p.status, WAIT_CLUSTER_PRODUCER, int(blockIdx.y), kb);
        for (int i = (issued > S ? issued - S : 0); i < issued; ++i) mbar_wait(&full_bar[i % S], uint32_t(i / S) & 1u, p.wait_limit);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t idesc = make_idesc_bf16(GEMM_BM, BN, A_MN, B_MN);
      const uint64_t dA = A_MN ? make_smem_desc(smem_u32(smem), 8192, 1024) : make_smem_desc(smem_u32(smem), 16, 1024);
      const uint64_t dB = B_MN ? make_smem_desc(smem_u32(smem) + GEMM_A_BYTES, 8192, 1024)
                               : make_smem_desc(smem_u32(smem) + GEMM_A_BYTES, 16, 1024);
      const uint32_t dA_hi = uint32_t(dA >> 32), dB_hi = uint32_t(dB >> 32);
      constexpr uint32_t stepA = (A_MN ? 2048 : 32) >> 4, stepB = (B_MN ? 2048 : 32) >> 4;
      uint32_t s = 0, ph = 0;
      bool ok = true;
      int kb = 0;
#pragma unroll 1
      for (int g = 0; g < SEGS && ok; ++g) {
        const uint32_t tacc = tmem_base + uint32_t(g * BN);
        const int end = SEGS == 1 ? num_kb : kb + num_kb / SEGS + (g < num_kb % SEGS ? 1 : 0);    // (the first parts take one more)
        uint32_t acc = 0;
        for (; kb < end; ++kb) {
          ok = mbar_wait_addr(full0 + 8u * s, ph, p.wait_limit);
          if (!ok) break;
          tc_fence_after();
          const uint32_t off = s * uint32_t(SM::STAGE_BYTES >> 4);
#pragma unroll
          for (int j = 0; j < GEMM_BK / 16; ++j) {
            umma_f16_lohi(tacc, uint32_t(dA) + off + j * stepA, dA_hi, uint32_t(dB) + off + j * stepB, dB_hi, idesc, acc);
            acc = 1;
          }
          umma_commit_addr(empty0 + 8u * s);
          if (++s == uint32_t(S)) { s = 0; ph ^= 1u; }
        }
      }
      umma_commit(acc_bar);
      if (!ok) report_expired(p.status, WAIT_CLUSTER_MMA, int(blockIdx.y), kb);
    }
  } else {
    const int q = warp & 3;
    if (warp == 2 && lane == 0) {
      // what the ring does not reach yet is asked into L2 meanwhile (the weights come from HBM on a first read)
      const int ahead = min(num_kb, S + 16);
      for (int kb = S; kb < ahead; ++kb) {
        const int kk = (kb0 + kb) * GEMM_BK;
        if (B_MN) {
#pragma unroll
          for (int c = 0; c < BN / 64; ++c) tma_prefetch_l2_2d(&tmB, tm.n0 + c * 64, kk);
        } else {
          tma_prefetch_l2_2d(&tmB, kk, tm.n0);
        }
      }
    }
    __syncwarp();
    bool ok = mbar_wait(acc_bar, 0, p.wait_limit);
    ok = __all_sync(0xffffffffu, ok);
    if (!ok && lane == 0) report_expired(p.status, WAIT_CLUSTER_EPILOGUE, int(blockIdx.y), -1);
    tc_fence_after();
    float* row = reinterpret_cast<float*>(smem) + (q * 32 + lane) * gemmc_part_pitch(BN);
    if (ok && tm.m0 + q * 32 < p.M) {
#pragma unroll
      for (int c = 0; c < BN / 32; ++c) {
        uint32_t r[32];
        tmem_ld_32x32(tmem_base + (uint32_t(q * 32) << 16) + uint32_t(c * 32), r);
        tmem_ld_wait();
#pragma unroll
        for (int s = 1; s < SEGS; ++s) {
          uint32_t t[32];
          tmem_ld_32x32(tmem_base + (uint32_t(q * 32) << 16) + uint32_t(s * BN + c * 32), t);
          tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 32; ++i) r[i] = __float_as_uint(__uint_as_float(r[i]) + __uint_as_float(t[i]));
        }
#pragma unroll
        for (int g = 0; g < 8; ++g)
          *reinterpret_cast<uint4*>(row + c * 32 + g * 4) = make_uint4(r[4 * g], r[4 * g + 1], r[4 * g + 2], r[4 * g + 3]);
      }
    }
  }
  __syncwarp();
  tc_fence_before();
  cluster_sync_all();                     // every partial tile of the cluster is in shared memory
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, BN * SEGS);
    if (lane == 0) tmem_note_freed(TK_GEMM, BN * SEGS);
  }
  const uint32_t part = smem_u32(smem);
  if constexpr (ONE) {
    gemmc_reduce_store<BN, MODE, 1>(p, tm, part, rank);
    return;
  }
  switch (C) {
    case 2: gemmc_reduce_store<BN, MODE, 2>(p, tm, part, rank); break;
    case 4: gemmc_reduce_store<BN, MODE, 4>(p, tm, part, rank); break;
    default: gemmc_reduce_store<BN, MODE, 8>(p, tm, part, rank); break;
  }
  __syncwarp();
  cluster_sync_all();                     // shared memory outlives the other CTAs' reads
}

}  // namespace lp
