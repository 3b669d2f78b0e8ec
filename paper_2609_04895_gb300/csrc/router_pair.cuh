// Router heads for N = 128 on CTA pairs (tcgen05 cta_group::2).
//
// router_gemm.cuh's kernel gives an SM a 128-row hidden tile and all H * 128
// weight rows of each K block, 64 KB for three heads and so three stages.  A
// pair runs M = 256 MMAs: each CTA holds its own hidden tile and half of the
// weight rows, 40 KB a K block for the same flops, and the even CTA issues the
// MMAs into both CTAs' TMEM.
//
// With three heads the accumulator takes 384 of the 512 TMEM columns and cannot
// be doubled, so what counts is how soon the epilogue has read it: eight warps
// take the heads in two groups, alternately, so the third head is read when the
// first is done, not the second.
//
// What bounds it: 24 streams x 500 tokens x 48 layers, d = 2048 (2.4 GB of
// hidden states read, 0.9 GB of scores written, 0.9 TFLOP) take 741 us with one
// CTA a tile and 701 on pairs (4.6 TB/s); without the stores 579, without the
// epilogue 533, the MMAs alone 480 at the cuBLAS rate.  d = 4096: 799 and 719.
//
// Warps (320 threads): 0 TMA producer, 1 TMEM owner and (even CTA) MMA issuer,
// 2..9 epilogue (warp w reads TMEM lanes 32 * (w % 4) .. + 31; group (w - 2) / 4).
#pragma once

#include "router_gemm.cuh"

namespace crc {

template <int H>
struct RouterPairCfg {
    static constexpr int NH = 128;
    using RC = RouterCfg<NH, H>;
    static constexpr int NACC = RC::NACC;
    static constexpr int W_ROWS = RC::NCH / 2;                 // this CTA's rows of one MMA
    static constexpr int STAGE_BYTES = RC::A_BYTES + RC::NMMA * W_ROWS * RC::BK * 2;
    static constexpr uint32_t IDESC = idesc_bf16_f32(256, RC::NCH);
    static constexpr int EPI_WARPS = 8;
    static constexpr int STAGING_BYTES = EPI_WARPS * 2 * 4096;
    static constexpr int STAGES = imin(8, (232448 - 1024 - 256 - STAGING_BYTES) / STAGE_BYTES);
    static constexpr int SMEM_BYTES = 1024 + STAGES * STAGE_BYTES + STAGING_BYTES + 256;
    static constexpr int THREADS = 32 * (2 + EPI_WARPS);
    // arrivals that hand an accumulator back: every head's four warps, both CTAs
    static constexpr int RELEASES = 2 * H * 4;
    static_assert(STAGES >= 3 && STAGE_BYTES % 1024 == 0 && (W_ROWS * 128) % 1024 == 0, "stages");
};

struct RouterPairArgs {
    RouterArgs r;
    int pairs_per_layer, num_pairs;     // tiles 2j and 2j + 1 of a layer; the last may be single
};

template <int H>
__global__ void __launch_bounds__(RouterPairCfg<H>::THREADS, 1)
    router_pair_kernel(const __grid_constant__ CUtensorMap tmap_h,
                       const __grid_constant__ CUtensorMap tmap_w,
                       const __grid_constant__ CUtensorMap tmap_s, RouterPairArgs pa) {
    using Cfg = RouterPairCfg<H>;
    using RC = typename Cfg::RC;
    constexpr int NH = Cfg::NH, NACC = Cfg::NACC;
    const RouterArgs& a = pa.r;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* staging = smem + Cfg::STAGES * Cfg::STAGE_BYTES;
    uint64_t* full_bar = reinterpret_cast<uint64_t*>(staging + Cfg::STAGING_BYTES);
    uint64_t* empty_bar = full_bar + Cfg::STAGES;
    uint64_t* tfull_bar = empty_bar + Cfg::STAGES;
    uint64_t* tempty_bar = tfull_bar + NACC;
    uint64_t* drain_bar = tempty_bar + NACC;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain_bar + 1);

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const bool leader = rank == 0u;
    const int first = (int)blockIdx.x >> 1, step = (int)gridDim.x >> 1;   // pairs of this cluster
    const int tiles_per_layer = a.n_sb * a.n_tb;

    if (threadIdx.x == 0) {
        for (int s = 0; s < Cfg::STAGES; ++s) {
            mbar_init(&full_bar[s], 1);
            mbar_init(&empty_bar[s], 1);
        }
        for (int s = 0; s < NACC; ++s) {
            mbar_init(&tfull_bar[s], 1);
            mbar_init(&tempty_bar[s], Cfg::RELEASES);
        }
        mbar_init(drain_bar, 1);
        fence_mbar_init();
        tma_prefetch_desc(&tmap_h);
        tma_prefetch_desc(&tmap_w);
        tma_prefetch_desc(&tmap_s);
    }
    if (warp == 1) {
        tmem_alloc_pair(tmem_slot, RC::TMEM_COLS);
        tmem_relinquish_pair();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();                     // the peer's barriers exist before any remote use
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    if (warp == 0) {
        // ------------------------------------------------------------ TMA
        if (lane == 0) {
            const uint64_t pol_h = l2_evict_first_policy();
            const uint64_t pol_w = l2_evict_last_policy();
            // both CTAs' loads of a stage complete on the even CTA's barrier
            const uint32_t lead_full = cluster_map(&full_bar[0], 0u);
            int stage = 0, issued = 0, failed = 0;
            uint32_t phase = 0;
            for (int q = first; q < pa.num_pairs && !failed; q += step) {
                const int l = q / pa.pairs_per_layer;
                const int r = 2 * (q % pa.pairs_per_layer) + (int)rank;
                const int sb = r / a.n_tb, tb = r % a.n_tb;   // past the layer: rows out of range, zeros
                for (int kb = 0; kb < a.kblocks; ++kb) {
                    if (!mbar_wait_cluster(&empty_bar[stage], phase ^ 1)) {
                        latch_error(a.err, CRC_ETIMEOUT);
                        failed = 1;
                        break;
                    }
                    uint8_t* sa = smem + stage * Cfg::STAGE_BYTES;
                    uint8_t* sw = sa + RC::A_BYTES;
                    if (leader) mbar_arrive_expect_tx(&full_bar[stage], 2 * Cfg::STAGE_BYTES);
                    const uint32_t fb = lead_full + (uint32_t)(stage * 8);
                    tma_load_4d_pair(sa, &tmap_h, fb, kb * RC::BK, l, a.t_begin + tb * a.TB,
                                     sb * a.SB, pol_h);
#pragma unroll
                    for (int c = 0; c < RC::NMMA; ++c)
                        tma_load_3d_pair(sw + c * Cfg::W_ROWS * 128, &tmap_w, fb, kb * RC::BK,
                                         c * RC::NCH + (int)rank * Cfg::W_ROWS, l, pol_w);
                    ++issued;
                    if (++stage == Cfg::STAGES) {
                        stage = 0;
                        phase ^= 1;
                    }
                }
            }
            // Never leave with copies in flight (the even CTA's barriers see both
            // CTAs' loads; the odd one stays for the final cluster barrier).
            int s = stage;
            uint32_t ph = phase;
            for (int k = 0; k < (leader ? imin(issued, Cfg::STAGES) : 0); ++k) {
                if (--s < 0) {
                    s = Cfg::STAGES - 1;
                    ph ^= 1;
                }
                if (!mbar_wait_cluster(&full_bar[s], ph)) latch_error(a.err, CRC_ETIMEOUT);
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA
        if (lane == 0 && leader) {
            int stage = 0, acc = 0, failed = 0;
            uint32_t phase = 0, acc_phase = 0;
            for (int q = first; q < pa.num_pairs && !failed; q += step) {
                if (!mbar_wait_cluster(&tempty_bar[acc], acc_phase ^ 1)) {
                    latch_error(a.err, CRC_ETIMEOUT);
                    break;
                }
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + (uint32_t)(acc * RC::ACC_COLS);
                for (int kb = 0; kb < a.kblocks; ++kb) {
                    if (!mbar_wait_cluster(&full_bar[stage], phase)) {
                        latch_error(a.err, CRC_ETIMEOUT);
                        failed = 1;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t sa = smem_u32(smem + stage * Cfg::STAGE_BYTES);
                    const uint32_t sw = sa + RC::A_BYTES;
#pragma unroll
                    for (int kk = 0; kk < RC::BK / 16; ++kk) {
                        const uint64_t adesc = sw128_kmajor_desc(sa + kk * 32);
#pragma unroll
                        for (int c = 0; c < RC::NMMA; ++c)
                            umma_bf16_pair(d_tmem + c * RC::NCH, adesc,
                                           sw128_kmajor_desc(sw + c * Cfg::W_ROWS * 128 + kk * 32),
                                           Cfg::IDESC, (kb | kk) != 0);
                    }
                    umma_commit_pair(&empty_bar[stage]);
                    if (++stage == Cfg::STAGES) {
                        stage = 0;
                        phase ^= 1;
                    }
                }
                if (failed) break;
                umma_commit_pair(&tfull_bar[acc]);
                if (NACC == 2) {
                    acc ^= 1;
                    if (acc == 0) acc_phase ^= 1;
                } else {
                    acc_phase ^= 1;
                }
            }
            umma_commit_pair_local(drain_bar);
            if (!mbar_wait(drain_bar, 0)) latch_error(a.err, CRC_ETIMEOUT);
        }
    } else {
        // ------------------------------------------------------------ epilogue
        const int quarter = warp & 3;
        const int group = (warp - 2) >> 2;
        uint8_t* my_stage = staging + (warp - 2) * 2 * 4096;
        const uint32_t tempty_lead = cluster_map(&tempty_bar[0], 0u);
        int buf = 0, acc = 0, turn = group;      // turn: this group's next head, counted from here
        uint32_t acc_phase = 0;
        for (int q = first; q < pa.num_pairs; q += step) {
            if (!mbar_wait_cluster(&tfull_bar[acc], acc_phase)) {
                latch_error(a.err, CRC_ETIMEOUT);
                break;
            }
            tc_fence_after();
            const int l = q / pa.pairs_per_layer;
            const int r = 2 * (q % pa.pairs_per_layer) + (int)rank;
            const int sb = r / a.n_tb, tb = r % a.n_tb;
            const bool real = r < tiles_per_layer &&
                              CRC_IN_BOUNDS(l < a.L && sb < a.n_sb && tb < a.n_tb, a.err);
            const int row0 = quarter * 32;
            const int str0 = sb * a.SB + row0 / a.TB;
            const int tok0 = tb * a.TB + row0 % a.TB;
            const uint32_t tbase =
                tmem_base + (uint32_t)(acc * RC::ACC_COLS) + ((uint32_t)(quarter * 32) << 16);
            int h = turn;
#pragma unroll 1
            for (; h < H; h += 2) {
                float z[NH];
#pragma unroll
                for (int c = 0; c < NH / 32; ++c)
                    tmem_ld32(tbase + (uint32_t)(h * NH + c * 32), z + 32 * c);
                tmem_ld_wait();
#pragma unroll
                for (int c = 0; c < NH / 16; ++c) pin16(z + 16 * c);
                tc_fence_before();                     // this head is read
                __syncwarp();
                if (lane == 0) {
                    if (leader)
                        mbar_arrive(&tempty_bar[acc]);
                    else
                        mbar_arrive_remote(tempty_lead + (uint32_t)(acc * 8));
                }
                if (!real) continue;
                // (kblocks is never 0.  The branch keeps the softmax a block of its
                // own: scheduled together with the loads and stores around it, it
                // does not fit ten warps' 168 registers and spills, 752 instead
                // of 701 us.)
                if (a.kblocks > 0) head_softmax<NH>(z);
#pragma unroll
                for (int c = 0; c < NH / 32; ++c) {
                    uint8_t* sbuf = my_stage + buf * 4096;
                    buf ^= 1;
                    if (lane == 0) bulk_wait_read<1>();   // the store that used sbuf is done
                    __syncwarp();
                    float4* dst = reinterpret_cast<float4*>(sbuf + lane * 128);
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        dst[j ^ (lane & 7)] =
                            make_float4(z[32 * c + 4 * j], z[32 * c + 4 * j + 1],
                                        z[32 * c + 4 * j + 2], z[32 * c + 4 * j + 3]);
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0) {
                        tma_store_5d(&tmap_s, sbuf, c * 32, h, l, tok0, str0);
                        bulk_commit();
                    }
                }
            }
            turn = h - H;
            if (NACC == 2) {
                acc ^= 1;
                if (acc == 0) acc_phase ^= 1;
            } else {
                acc_phase ^= 1;
            }
        }
        if (lane == 0) bulk_wait<0>();                 // every store has landed
    }

    tc_fence_before();
    __syncthreads();
    // neither CTA leaves (or frees TMEM) while the other may still arrive on its
    // barriers or have MMAs write its TMEM
    cluster_sync();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, RC::TMEM_COLS);
    }
}

}  // namespace crc
