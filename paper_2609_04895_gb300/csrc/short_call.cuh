// Route-and-cache for short calls (one decoded token, a few draft tokens, a
// small chunk): one cluster of CTAs per (layer, stream group), nothing shared
// between clusters.
//
// The persistent fused kernel (fused.cuh) gives a tile all three heads of one
// layer, so a one-token call of the Qwen3 shape runs 48 tiles on 152 SMs, and
// every chain then waits for the tile of the layer before it (p^S of the
// predecessor) through the record ring in global memory.  Here the CTAs of a
// cluster take one head each,
//     rank 0: R of layer l,   rank 1: T of layer l,   rank 2: S of layer l - 1
// (S of layer L - 1 for l = 0: the predecessor of token t is token t - 1
// there, and the last token's row is the carry for the next call), over all T
// tokens of the group's streams, which fit the 128 rows of one tile.  So a
// cluster holds everything its chains need: the probabilities stay in the
// three CTAs' shared memory, the scan warps read them there (distributed
// shared memory) after one cluster barrier, and there is no ring, no control
// block to clear and no cooperative launch.  Each weight row is read by one
// CTA per stream group, each hidden row by three (twice from L2).
//
// What bounds it: one token of 64 streams of the Qwen3 shape takes 31 us (the
// persistent kernel 56, after clearing its control block): 2.5 us to the first
// data, 13.5 us for the GEMM, which reads 88 MB at 6.5 TB/s, then softmax,
// Top-K sets, one step of two chains a warp and the cluster barriers, a
// microsecond or two each.  With more tokens it is the chains' steps, 0.75 us
// each (24 tokens of 13 streams: 91 -> 63 us); the rows of a step are asked for
// one step ahead with nothing in between that waits for them (0.91 us when the
// normalisers were multiplied in at the load), and the trace's words are
// gathered after the chains (1.05 us when they were gathered in the step).
//
// Per CTA: warp 0 issues the TMA loads, warp 1 owns TMEM and issues the MMAs;
// then warps 0..7 take the softmax (two threads a tile row, half a head each),
// and after the cluster barrier all warps take the Top-K sets of the rows of
// this CTA's chains (streams rank, rank + H, ... of the group), then the
// chains.  The arithmetic is that of the router and fused kernels in the same
// order, so the results are theirs bit for bit.
#pragma once

#include "cache_scan.cuh"
#include "router_gemm.cuh"

namespace crc {

constexpr int kShortWarps = 12;      // at most; 8 when more CTAs than 2 an SM want in
constexpr int kShortMaxStages = 12;

template <int NH>
struct ShortCfg {
    static constexpr int BK = 64;
    static constexpr int W_BYTES = NH * BK * 2;               // weight rows of one head
    static constexpr int TMEM_COLS = pow2ceil_i(imax(32, NH));
    static constexpr int CW = NH < 32 ? NH : 32;              // TMEM columns per load
    static constexpr int NCHK = NH / CW;
    static constexpr int NW = (NH + 31) / 32;
    static constexpr int ROW_FLOATS = NH + 4;                 // 16 bytes of padding: no bank conflicts
    static constexpr uint32_t IDESC = idesc_bf16_f32(128, NH);
    // barriers, TMEM slot, fail flag; the two halves' maxima and sums
    static constexpr int TAIL_BYTES = 256 + 128 * 4 * 4;
    static constexpr int MAX_THREADS = 32 * kShortWarps;
};

struct ShortArgs {
    uint8_t* state;
    int B, L, N, K, C, R, T;
    int SB, n_bg;           // a cluster's tile: SB streams x T tokens <= 128 rows
    int kblocks, stages;
    int a_bytes;            // bytes of a hidden box: SB * T rows of 128
    int stage_bytes;        // hidden box rounded up to 1024, weight box
    int sel_at, tr_at, tail;   // offsets of the Top-K bytes, of the traced sets and of the tail
    uint8_t* tr_miss;       // optional trace, as in FusedArgs
    uint8_t* tr_pro;
    uint32_t* tr_mid;
    uint32_t* tr_after;
    uint32_t* tr_sel;
};

// Descending sort of a lane's V keys (V = 1, 2, 4, 8): Batcher's odd-even
// merge sort, 1, 5 and 19 compare-exchanges.
template <int V>
__device__ __forceinline__ void sort_desc_keys(uint32_t (&a)[V]) {
#pragma unroll
    for (int p = 1; p < V; p <<= 1) {
#pragma unroll
        for (int k = p; k >= 1; k >>= 1) {
#pragma unroll
            for (int j = k % p; j + k < V; j += 2 * k) {
#pragma unroll
                for (int i = 0; i < k; ++i) {
                    const int x = i + j, y = i + j + k;
                    if (y < V && x / (2 * p) == y / (2 * p)) {
                        const uint32_t hi = umax(a[x], a[y]), lo = umin(a[x], a[y]);
                        a[x] = hi;
                        a[y] = lo;
                    }
                }
            }
        }
    }
}

// The Top-K sets of G rows held by the warp (V keys a lane, 0 in invalid slots).  A lane sorts its keys; K rounds pop
// the largest head over the warp (one redux.sync, then the lane whose head it
// is moves up its list), the rows' rounds interleaved so their latencies
// overlap.  Exactly K keys at or above the last popped one prove that those
// are the set; any other count (equal keys, or fewer than K above 0) goes to
// topk_ties.
template <int V, int G>
__device__ __forceinline__ void topk_sets(const uint32_t (&row)[G][V], uint32_t valid, int lane,
                                          int K, uint32_t (&set)[G]) {
    uint32_t h[G][V], th[G];
#pragma unroll
    for (int g = 0; g < G; ++g) {
#pragma unroll
        for (int v = 0; v < V; ++v) h[g][v] = row[g][v];
        sort_desc_keys<V>(h[g]);
        th[g] = 0u;
    }
#pragma unroll 1
    for (int k = 0; k < K; ++k) {
#pragma unroll
        for (int g = 0; g < G; ++g) th[g] = __reduce_max_sync(kFull, h[g][0]);
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const bool mine = h[g][0] == th[g];
#pragma unroll
            for (int v = 0; v + 1 < V; ++v) h[g][v] = mine ? h[g][v + 1] : h[g][v];
            h[g][V - 1] = mine ? 0u : h[g][V - 1];
        }
    }
    uint32_t c = 0u;                           // two counts of at most 256 to a reduction
    static_assert(G <= 2, "counts packed by two");
#pragma unroll
    for (int g = 0; g < G; ++g) {
        set[g] = 0u;
#pragma unroll
        for (int v = 0; v < V; ++v) set[g] |= row[g][v] >= th[g] ? 1u << v : 0u;
        c += (uint32_t)__popc(set[g]) << (16 * g);
    }
    c = __reduce_add_sync(kFull, c);
#pragma unroll
    for (int g = 0; g < G; ++g) {
        if (((c >> (16 * g)) & 0xffffu) == (uint32_t)K) continue;
        Keys<V> key;
#pragma unroll
        for (int v = 0; v < V; ++v) key.k[v] = row[g][v];
        set[g] = topk_ties<V>(key, valid, lane, K);
    }
}

// V floats at a shared::cluster address (16-byte aligned for V >= 4).
template <int V>
__device__ __forceinline__ void dsm_vec(uint32_t addr, float (&out)[V]) {
    if constexpr (V == 4) {
        asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(out[0]), "=f"(out[1]), "=f"(out[2]), "=f"(out[3])
                     : "r"(addr));
    } else if constexpr (V == 2) {
        asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];"
                     : "=f"(out[0]), "=f"(out[1])
                     : "r"(addr));
    } else {
        static_assert(V == 1, "experts per lane");
        asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(out[0]) : "r"(addr));
    }
}
__device__ __forceinline__ uint32_t dsm_u32(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}

// TRACED: compiled with the trace writes (any trace array given).
template <int NH, int V, bool ALL_VALID, bool TRACED>
__global__ void __launch_bounds__(ShortCfg<NH>::MAX_THREADS, 2)
    short_call_kernel(const __grid_constant__ CUtensorMap tmap_h,
                      const __grid_constant__ CUtensorMap tmap_w, ShortArgs a) {
    using Cfg = ShortCfg<NH>;
    constexpr int CW = Cfg::CW, NW = Cfg::NW;
    constexpr int ROW = Cfg::ROW_FLOATS;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* full_bar = reinterpret_cast<uint64_t*>(smem + a.tail);
    uint64_t* empty_bar = full_bar + kShortMaxStages;
    uint64_t* tfull_bar = empty_bar + kShortMaxStages;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tfull_bar + 1);
    uint32_t* fail = tmem_slot + 1;
    float* half_max = reinterpret_cast<float*>(smem + a.tail + 256);   // [2][128]
    float* half_sum = half_max + 256;                                  // [2][128]
    // after the GEMM the stages hold this head's probabilities, [rows][ROW], and behind
    // them the Top-K bits of this CTA's chains, one byte a lane, [rows][32], and
    // in traced calls the cache before (low half) and after the update likewise,
    // and the rows' misses and proactive loads
    float* probs = reinterpret_cast<float*>(smem);
    uint8_t* sel_s = smem + a.sel_at;
    uint8_t* sets_s = smem + a.tr_at;

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int warps = (int)blockDim.x >> 5;
    const int rank = (int)cluster_ctarank();
    const int H = a.R > 0 ? 3 : 2;
    const int group = (int)blockIdx.x / H;
    const int l = group / a.n_bg, bg = group % a.n_bg;
    const int b0 = bg * a.SB;                                   // the group's first stream
    const int n_str = imin(a.SB, a.B - b0);
    const int n_own = (n_str - rank + H - 1) / H;               // chains of this CTA
    const int lw = rank == 2 ? (l > 0 ? l - 1 : a.L - 1) : l;   // layer of this CTA's head
    StateHeader* hdr = reinterpret_cast<StateHeader*>(a.state);
    uint32_t* err = &hdr->error;
    const bool in_bounds = CRC_IN_BOUNDS(
        l < a.L && b0 < a.B && lw < a.L && n_str * a.T <= 128 && n_str * a.T * ROW * 4 <= a.sel_at &&
            n_own * a.T * 32 <= a.tr_at - a.sel_at &&
            (!TRACED || a.tr_at + n_own * a.T * 34 <= a.tail) && a.tr_at <= a.tail &&
            a.stages * a.stage_bytes <= a.tail,
        err);
    auto timed_out = [&] {
        latch_error(err, CRC_ETIMEOUT);
        atomicExch(fail, 1u);
        atomicExch(&hdr->aborted, 1u);
    };

    if (warp == 0) {
        // ------------------------------------------------------------ TMA
        // Before anything else: the loads need the barriers alone, and the
        // weights' first blocks come from DRAM.
        if (lane == 0) {
            for (int s = 0; s < a.stages; ++s) {
                mbar_init(&full_bar[s], 1);
                mbar_init(&empty_bar[s], 1);
            }
            mbar_init(tfull_bar, 1);
            *fail = 0u;
            fence_mbar_init();
        }
        __syncwarp();
    }
    const uint64_t pol_h = l2_evict_first_policy();
    const uint64_t pol_w = l2_evict_last_policy();
    auto load_stage = [&](int kb, int stage) {
        uint8_t* sa = smem + stage * a.stage_bytes;
        uint8_t* sw = sa + (a.stage_bytes - Cfg::W_BYTES);
        mbar_arrive_expect_tx(&full_bar[stage], (uint32_t)(a.a_bytes + Cfg::W_BYTES));
        tma_load_3d(sw, &tmap_w, &full_bar[stage], kb * Cfg::BK, rank * NH, lw, pol_w);
        tma_load_4d(sa, &tmap_h, &full_bar[stage], kb * Cfg::BK, lw, 0, b0, pol_h);
    };
    if (warp == 0 && lane == 0 && in_bounds)
        for (int kb = 0; kb < imin(a.stages, a.kblocks); ++kb) load_stage(kb, kb);
    if (warp == 1) {
        tmem_alloc(tmem_slot, Cfg::TMEM_COLS);
        tmem_relinquish();
    }
    const bool hdr_ok = hdr->magic == kStateMagic && hdr->L == a.L && hdr->N == a.N &&
                        hdr->K == a.K && hdr->C == a.C && hdr->R == a.R && hdr->B == a.B &&
                        hdr->policy == 0u;
    const int64_t t0g = hdr->t_next;
    const uint32_t parity = hdr->parity;
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    if (warp == 0) {
        if (lane == 0 && in_bounds) {
            int stage = 0, kb = a.stages;
            uint32_t phase = 0;                                // phase of the stages' next use
            for (; kb < a.kblocks; ++kb) {
                if (!mbar_wait(&empty_bar[stage], phase)) {
                    timed_out();
                    break;
                }
                load_stage(kb, stage);
                if (++stage == a.stages) {
                    stage = 0;
                    phase ^= 1;
                }
            }
            // never leave with copies in flight: wait for every issued stage to
            // land (use u of a stage completes its full barrier's phase u)
            const int issued = imin(kb, a.kblocks);
            for (int k = issued - imin(issued, a.stages); k < issued; ++k)
                if (!mbar_wait(&full_bar[k % a.stages], (uint32_t)(k / a.stages) & 1u)) timed_out();
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA
        if (lane == 0 && in_bounds) {
            int stage = 0;
            uint32_t phase = 0;
            for (int kb = 0; kb < a.kblocks; ++kb) {
                if (!mbar_wait(&full_bar[stage], phase)) {
                    timed_out();
                    break;
                }
                tc_fence_after();
                // rows past the hidden box read whatever follows in shared
                // memory: they fill accumulator rows nobody reads
                const uint32_t sa = smem_u32(smem + stage * a.stage_bytes);
                const uint32_t sw = sa + (uint32_t)(a.stage_bytes - Cfg::W_BYTES);
#pragma unroll
                for (int kk = 0; kk < Cfg::BK / 16; ++kk)
                    umma_bf16(tmem_base, sw128_kmajor_desc(sa + kk * 32),
                              sw128_kmajor_desc(sw + kk * 32), Cfg::IDESC, (kb | kk) != 0);
                umma_commit(&empty_bar[stage]);
                if (++stage == a.stages) {
                    stage = 0;
                    phase ^= 1;
                }
            }
            umma_commit(tfull_bar);
        }
        __syncwarp();
    }

    // ---------------------------------------------------------------- chains
    // Chain j of this CTA is stream rank + H * j of the group; a warp takes
    // j = wj, wj + warps, ...  Its state is fetched one chain ahead, the first
    // while the GEMM runs.
    const StateLayout lay = state_layout(a.B, a.L, a.N);
    ChainState* chains = reinterpret_cast<ChainState*>(a.state + lay.chains);
    float* retention = reinterpret_cast<float*>(a.state + lay.retention);
    float* carry = reinterpret_cast<float*>(a.state + lay.carry);
    const int N = a.N, L = a.L, T = a.T;
    uint32_t valid = 0u;
#pragma unroll
    for (int v = 0; v < V; ++v)
        if (lane * V + v < N) valid |= 1u << v;
    const bool has = valid != 0u;
    const uint32_t e0 = (uint32_t)lane * V;
    const bool want_s = a.R > 0;
    const bool runs = hdr_ok && in_bounds && CRC_IN_BOUNDS(parity < 2u, err);
    struct Loaded {
        uint32_t bits;
        Vec<V> aT;
        uint64_t hits, misses, pro;
    };
    auto load_chain = [&](int j) {
        Loaded q;
        const int chain = (b0 + rank + H * j) * L + l;
        if (!CRC_IN_BOUNDS(b0 + rank + H * j < a.B, err)) return Loaded{};
        const ChainState& cs = chains[chain];
        q.bits = lane_bits<V>(cs.bits, lane, N);
        q.aT = load_vec<V>(retention + (size_t)chain * N + e0, has);
        q.hits = cs.hits;
        q.misses = cs.misses;
        q.pro = cs.proactive;
        return q;
    };
    const int wj = warps - 1 - warp;
    Loaded next = {};
    if (runs && wj < n_own) next = load_chain(wj);

    if (warp < 8) {
        // ------------------------------------------------------------ softmax
        // Two threads a row: `half` of the head's columns each (the halves the
        // head's sum is defined over), maxima and sums exchanged.
        const int quarter = warp & 3, half = warp >> 2;
        const int row = quarter * 32 + lane;
        const bool live = in_bounds && quarter * 32 < n_str * T;
        constexpr int HW = NH / 2;                              // columns of a half
        constexpr int HC = HW < CW ? HW : CW;                   // columns of a load
        if (live) {
            if (!mbar_wait(tfull_bar, 0)) timed_out();
            tc_fence_after();
            const uint32_t tbase =
                tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(half * HW);
            auto load = [&](int c, float* z) {
                if constexpr (HC == 32) tmem_ld32(tbase + (uint32_t)c, z);
                else if constexpr (HC == 16) tmem_ld16f(tbase + (uint32_t)c, z);
                else tmem_ld8f(tbase + (uint32_t)c, z);
                tmem_ld_wait();
                if constexpr (HC >= 16) {
#pragma unroll
                    for (int i = 0; i < HC; i += 16) pin16(z + i);
                } else {
                    pin8(z);
                }
            };
            float z[HC];
            float m = -INFINITY;
#pragma unroll
            for (int c = 0; c < HW; c += HC) {
                load(c, z);
                m = max_of<HC>(z, m);
            }
            half_max[half * 128 + row] = m;
            named_sync(1 + quarter, 64);                        // the row quarter's two warps
            m = fmaxf(m, half_max[(half ^ 1) * 128 + row]);
            HeadExp x;
            x.init(m);
            float* out = probs + (size_t)row * ROW + half * HW;
            const bool wr = row < n_str * T;
#pragma unroll
            for (int c = 0; c < HW; c += HC) {
                load(c, z);
                x.template exp_in_place<HC>(z);
                if (wr) {
#pragma unroll
                    for (int q = 0; q < HC / 4; ++q)
                        *reinterpret_cast<float4*>(out + c + 4 * q) =
                            make_float4(z[4 * q], z[4 * q + 1], z[4 * q + 2], z[4 * q + 3]);
                }
            }
            half_sum[half * 128 + row] = x.part();
            named_sync(1 + quarter, 64);
            const float r = head_inv(half_sum[row], half_sum[128 + row]);
            if (wr) {
#pragma unroll
                for (int c = 0; c < HW; c += HC) {
                    float4* at = reinterpret_cast<float4*>(out + c);
#pragma unroll
                    for (int q = 0; q < HC / 4; ++q) {
                        const float4 f = at[q];
                        z[4 * q] = f.x;
                        z[4 * q + 1] = f.y;
                        z[4 * q + 2] = f.z;
                        z[4 * q + 3] = f.w;
                    }
                    scale_in_place<HC>(z, r);
#pragma unroll
                    for (int q = 0; q < HC / 4; ++q)
                        at[q] = make_float4(z[4 * q], z[4 * q + 1], z[4 * q + 2], z[4 * q + 3]);
                }
            }
        }
    }

    // every head's probabilities are in place in the cluster
    cluster_sync();
    const uint32_t fail_any = dsm_u32(cluster_map(fail, 0u)) | dsm_u32(cluster_map(fail, 1u)) |
                              (H == 3 ? dsm_u32(cluster_map(fail, 2u)) : 0u);
    const bool go = runs && fail_any == 0u;
    // this lane's part of row 0 of each head
    const uint32_t pR_at = cluster_map(probs, 0u) + e0 * 4u;
    const uint32_t pT_at = cluster_map(probs, 1u) + e0 * 4u;
    const uint32_t pS_at = H == 3 ? cluster_map(probs, 2u) + e0 * 4u : 0u;
    if (go) {
        // Top-K sets of this CTA's rows (chain j, token t) = j * T + t, two at a time
        const int rows = n_own * T;
        for (int i = 2 * warp; i < rows; i += 2 * warps) {
            uint32_t key[2][V], set[2];
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                const int ii = imin(i + g, rows - 1);
                const uint32_t r = (uint32_t)((rank + H * (ii / T)) * T + ii % T);
                float p[V];
#pragma unroll
                for (int v = 0; v < V; ++v) p[v] = 0.f;
                if (has) dsm_vec<V>(pR_at + r * (ROW * 4u), p);
#pragma unroll
                for (int v = 0; v < V; ++v) key[g][v] = __float_as_uint(p[v]);
            }
            topk_sets<V, 2>(key, valid, lane, a.K, set);
            sel_s[i * 32 + lane] = (uint8_t)set[0];
            if (i + 1 < rows) sel_s[(i + 1) * 32 + lane] = (uint8_t)set[1];
        }
    }
    __syncthreads();
    if (go) {
#pragma unroll 1
        for (int j = wj; j < n_own; j += warps) {
            const int si = rank + H * j;
            const int b = b0 + si;
            const int chain = b * L + l;
            const Loaded cur = next;
            ChainRegs<V> cr;
            cr.set_bits(cur.bits);
            cr.count = (int)__reduce_add_sync(kFull, (uint32_t)__popc(cur.bits));
#pragma unroll
            for (int v = 0; v < V; ++v) cr.aT[v] = cur.aT.v[v];
            cr.hits = cr.misses = cr.pro = 0u;
            const uint32_t r0 = (uint32_t)(si * T);
            // the rows of step t, asked for a step ahead: nothing here waits for them
            struct In {
                float R[V], T[V], S[V];
            };
            auto fetch = [&](int t, In& q) {
#pragma unroll
                for (int v = 0; v < V; ++v) q.R[v] = q.T[v] = q.S[v] = 0.f;
                if (!has) return;
                const uint32_t at = (r0 + (uint32_t)t) * (ROW * 4u);
                dsm_vec<V>(pR_at + at, q.R);
                dsm_vec<V>(pT_at + at, q.T);
                if (want_s && t0g + t >= 1) {
                    if (l > 0 || t > 0) {
                        dsm_vec<V>(pS_at + (l > 0 ? at : at - ROW * 4u), q.S);
                    } else {
                        const Vec<V> x =
                            load_vec<V>(carry + ((size_t)parity * a.B + b) * N + e0, true);
#pragma unroll
                        for (int v = 0; v < V; ++v) q.S[v] = x.v[v];
                    }
                }
            };
            In q, ahead;
            fetch(0, q);
            if (j + warps < n_own) next = load_chain(j + warps);
#pragma unroll 1
            for (int t = 0; t < T; ++t) {
                if (t + 1 < T) fetch(t + 1, ahead);
                float sT[V];
#pragma unroll
                for (int v = 0; v < V; ++v) sT[v] = __fadd_rn(q.R[v], q.T[v]);
                const uint32_t sel = sel_s[(j * T + t) * 32 + lane];
                Sel<V> s;
                sel_from_bits<V>(sel, s);
                const int i = j * T + t;
                int nD;
                uint32_t mid = 0u;
                const int pro = scan_apply<V, ALL_VALID>(
                    cr, sT, q.S, want_s && t0g + t >= 1, valid, lane, a.K, a.C, a.R, s, &nD,
                    [](Sel<V>&) {}, [&] { if (TRACED) mid = cr.bits(lane); });
                if constexpr (TRACED) {
                    sets_s[i * 32 + lane] = (uint8_t)(mid | (cr.bits(lane) << 4));
                    if (lane == 0)
                        *reinterpret_cast<uchar2*>(sets_s + n_own * T * 32 + i * 2) =
                            make_uchar2((unsigned char)nD, (unsigned char)pro);
                }
                (void)CRC_IN_BOUNDS((cr.bits(lane) & ~valid) == 0u && cr.count <= a.C, err);
                q = ahead;
            }
            // layer 0's cluster holds p^S of layer L - 1: its last token is the carry
            if (l == 0 && want_s && has) {
                float pl[V];
                dsm_vec<V>(pS_at + (r0 + (uint32_t)(T - 1)) * (ROW * 4u), pl);
                float* dst = carry + ((size_t)(parity ^ 1u) * a.B + b) * N + e0;
#pragma unroll
                for (int v = 0; v < V; ++v)
                    if (lane * V + v < N) dst[v] = pl[v];
            }
            ChainState& cs = chains[chain];
            store_cache_words<V>(cr.bits(lane), lane, N, cs.bits);
            if (has) {
#pragma unroll
                for (int v = 0; v < V; ++v)
                    if (lane * V + v < N) retention[(size_t)chain * N + e0 + v] = cr.aT[v];
            }
            if (lane == 0) {
                cs.hits = cur.hits + cr.hits;
                cs.misses = cur.misses + cr.misses;
                cs.proactive = cur.pro + cr.pro;
            }
        }
    }

    if constexpr (TRACED) {
        // the rows' trace, a row a warp (out of the chains' way: gathering the
        // sets' words there cost 0.4 us a token)
        __syncthreads();
        for (int i = warp; go && i < n_own * T; i += warps) {
            const int t = i % T;
            const int b = b0 + rank + H * (i / T);
            if (!CRC_IN_BOUNDS(b < a.B && l < L, err)) continue;
            const size_t unit = ((size_t)b * T + t) * L + l;
            const uint32_t sets = sets_s[i * 32 + lane], sel = sel_s[i * 32 + lane];
            if (a.tr_mid) store_cache_words<V>(sets & 15u, lane, N, a.tr_mid + unit * NW);
            if (a.tr_after) store_cache_words<V>(sets >> 4, lane, N, a.tr_after + unit * NW);
            if (a.tr_sel) store_cache_words<V>(sel, lane, N, a.tr_sel + unit * NW);
            if (lane < 2) {
                uint8_t* dst = lane == 0 ? a.tr_miss : a.tr_pro;
                if (dst) dst[unit] = sets_s[n_own * T * 32 + i * 2 + lane];
            }
        }
    }

    // no CTA leaves while another still reads its shared memory
    tc_fence_before();
    cluster_sync();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, Cfg::TMEM_COLS);
    }
    // the last CTA to finish advances the token counter and flips the carry slot
    if (threadIdx.x == 0) {
        if (!hdr_ok && blockIdx.x == 0) latch_error(err, CRC_ESTATE);
        __threadfence();
        const uint32_t prev = atomicAdd(&hdr->done, 1u);
        if (prev == gridDim.x - 1) {
            __threadfence();
            if (hdr_ok && *reinterpret_cast<volatile uint32_t*>(&hdr->aborted) == 0u) {
                hdr->t_next = t0g + a.T;
                hdr->parity = parity ^ 1u;
            }
            hdr->aborted = 0u;
            hdr->done = 0u;
            __threadfence();
        }
    }
}

}  // namespace crc
