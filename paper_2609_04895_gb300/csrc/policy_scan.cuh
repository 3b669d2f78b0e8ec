// Cache scans under the comparison policies of the paper's evaluation: the
// classical cache-update policies LRU, LFU and LRFU (lambda a multiple of
// 1/2; the paper uses 0.5) and the Spatio-only ablation (Algorithm 2's
// refinement on s^S = p^R_{t-1} + p^S_rho, LRU for demand misses; Sec. 4.3 and
// the appendix on ablations).  Same layout and reductions as the method's scan
// (cache_scan.cuh): one warp per (stream, layer) chain, lane i owns experts
// [iV, iV + V), priorities as ordered 32-bit keys.
//
// Readings (the paper names the policies and their references only):
//   - the classical policies only update the cache (no refinement, no
//     proactive load); each access demand-loads S \ C and, the cache being
//     full, evicts the member of C \ S with the lowest priority, ties to the
//     highest expert index, as Algorithm 1 does with s^T;
//   - LRU priority: the token of last use; LFU: the accesses that selected the
//     expert since it entered the cache; LRFU: CRF * F(t - t_last), the CRF
//     updated at each use to 1 + F(t - t_last) * CRF (1 on insertion), with
//     F(x) = 2^(-lambda x) computed in fp32 as 2^(-q) times fp32(2^(-1/2)) for
//     an odd number of halves, and 0 once q >= 126;
//   - Spatio-only: an expert its refinement loads counts as used at t.
#pragma once

#include "cache_scan.cuh"

namespace crc {

struct PolicyArgs {
    ScanArgs s;
    int policy;      // CRC_POLICY_*
    int lambda2;     // LRFU: lambda = lambda2 / 2
};

// F(dt) = 2^(-lambda dt) with lambda = lambda2 / 2.
__device__ __forceinline__ float lrfu_decay(int lambda2, uint32_t dt) {
    const uint32_t halves = (uint32_t)lambda2 * dt;
    const uint32_t q = halves >> 1;
    if (q >= 126u) return 0.f;
    float f = __uint_as_float((127u - q) << 23);                 // 2^-q, exact
    if (halves & 1u) f = __fmul_rn(f, 0.70710678118654752f);      // fp32(2^-1/2)
    return f;
}

// One access of the chain at token t under the policy POL (a CRC_POLICY_*
// value, fixed at compile time so that each policy's step carries only its
// own priority arithmetic).  aux: this lane's integer priorities (LRU,
// Spatio-only, LRFU: token of last use; LFU: count); cr.aT: the float ones
// (LRFU: CRF; Spatio-only: p^R of the previous token).
template <int V, bool ALL_VALID, int POL, class X>
__device__ __forceinline__ void policy_step(ChainRegs<V>& cr, uint32_t (&aux)[V],
                                            const float (&pR)[V], const float (&pS)[V],
                                            bool refine, uint32_t valid, int lane,
                                            const PolicyArgs& a, uint32_t t, Sel<V>& s,
                                            X exact_set, uint8_t* miss_out, uint8_t* pro_out) {
    const int K = a.s.K, C = a.s.C;
    int pro = 0, nD;
    bool in_s[V], was_in[V];                   // S, and the cache before the demand loads
    // the priority that evicts, as an ordered word
    auto word = [&](int v) {
        return POL == CRC_POLICY_LRFU ? __float_as_uint(__fmul_rn(
                                            cr.aT[v], lrfu_decay(a.lambda2, t - aux[v])))
                                      : aux[v];
    };
    if constexpr (V == 1) {
        if (POL == CRC_POLICY_SPATIO_LRU && refine) {
            const uint32_t before = cr.cache;
            pro = refine_mask(cr, pS[0], valid, lane, C, a.s.R);
            if (((cr.cache & ~before) >> lane) & 1u) aux[0] = t;
        }
        if (__popc(s.m) != K) exact_set(s);                      // scores tie at the threshold
        in_s[0] = ((s.m >> lane) & 1u) != 0u;
        was_in[0] = ((cr.cache >> lane) & 1u) != 0u;
        nD = __popc(s.m & ~cr.cache);
        const int over = cr.count + nD - C;
        update_mask(cr, over > 0 ? word(0) : 0u, s.m, over, lane);
        cr.count = over > 0 ? C : cr.count + nD;
    } else {
        uint32_t counts;
        if (POL == CRC_POLICY_SPATIO_LRU && refine) {
            float before[V];
#pragma unroll
            for (int v = 0; v < V; ++v) before[v] = cr.out[v];
            pro = scan_refine<V, ALL_VALID>(cr, pS, valid, lane, C, a.s.R, s, &counts);
            if (pro > 0) {
#pragma unroll
                for (int v = 0; v < V; ++v)
                    if (before[v] > cr.out[v]) aux[v] = t;           // came in
            }
        } else {
            counts = warp_count(__fadd_rn(miss_count<V>(cr, s), kCount0));
        }
        if ((counts >> 6) != (uint32_t)K) {                          // scores tie at the threshold
            exact_set(s);
            counts = warp_count(__fadd_rn(miss_count<V>(cr, s), kCount0));
        }
        nD = (int)(counts & 63u);
        // demand loads; a full cache evicts the lowest priorities outside S (they
        // do not change while the access inserts, and inserted experts are in S)
#pragma unroll
        for (int v = 0; v < V; ++v) {
            in_s[v] = s.s[v] != 0.f;
            was_in[v] = cr.out[v] == 0.f;
        }
        const int over = cr.count + nD - C;
        if (over > 0) {
            float key[V];
            // Integer priorities tie all the time (experts last used at the same
            // token), so while they fit (none exceeds the token index) the
            // expert's position from the end goes below them: distinct keys in the
            // same order, below 2^126 as bits of a float.
            if (POL != CRC_POLICY_LRFU && t < (1u << 22)) {
#pragma unroll
                for (int v = 0; v < V; ++v)
                    key[v] = __uint_as_float((aux[v] << 8) | (255u - (uint32_t)(lane * V + v)));
                update_cache<V, KeyTies::kNone>(cr, key, s, over, C - K, lane);
            } else {
                // (aux above 2^126's bits would need 2 billion tokens)
#pragma unroll
                for (int v = 0; v < V; ++v) key[v] = __uint_as_float(word(v));
                update_cache<V, KeyTies::kOften>(cr, key, s, over, C - K, lane);
            }
            cr.count = C;
        } else {
#pragma unroll
            for (int v = 0; v < V; ++v) cr.out[v] = __fmaf_rn(-s.s[v], cr.out[v], cr.out[v]);
            cr.count += nD;
        }
    }
    // the selected experts' priorities after the access
#pragma unroll
    for (int v = 0; v < V; ++v) {
        if (!in_s[v]) continue;
        const bool h = was_in[v];
        if constexpr (POL == CRC_POLICY_LFU) {
            aux[v] = h ? aux[v] + 1u : 1u;
        } else if constexpr (POL == CRC_POLICY_LRFU) {
            cr.aT[v] = h ? __fadd_rn(1.f, __fmul_rn(lrfu_decay(a.lambda2, t - aux[v]), cr.aT[v]))
                         : 1.f;
            aux[v] = t;
        } else {
            aux[v] = t;
        }
    }
    if constexpr (POL == CRC_POLICY_SPATIO_LRU) {
#pragma unroll
        for (int v = 0; v < V; ++v) cr.aT[v] = pR[v];            // p^R_{t-1} for the next access
    }
    cr.hits += (uint32_t)(K - nD);
    cr.misses += (uint32_t)nD;
    cr.pro += (uint32_t)pro;
    if (lane == 0) {
        if (miss_out) *miss_out = (uint8_t)nD;
        if (pro_out) *pro_out = (uint8_t)pro;
    }
}

template <int V, bool ALL_VALID, int KP, int POL>
__global__ void __launch_bounds__(32 * kScanWarps, (V >= 8 ? 12 : 24) / kScanWarps)
    cache_scan_policy_kernel(PolicyArgs pa) {
    const ScanArgs& a = pa.s;
    StateHeader* hdr = reinterpret_cast<StateHeader*>(a.state);
    const StateLayout lay = state_layout(a.B, a.L, a.N);
    ChainState* chains = reinterpret_cast<ChainState*>(a.state + lay.chains);
    float* val = reinterpret_cast<float*>(a.state + lay.retention);
    float* carry = reinterpret_cast<float*>(a.state + lay.carry);
    uint32_t* auxs = reinterpret_cast<uint32_t*>(a.state + lay.aux);

    const int lane = threadIdx.x & 31;
    const int chain = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const bool active = chain < a.B * a.L;
    // a state belongs to one policy: the one that first used it
    const bool hdr_ok = hdr->magic == kStateMagic && hdr->L == a.L && hdr->N == a.N &&
                        hdr->K == a.K && hdr->C == a.C && hdr->R == a.R && hdr->B == a.B &&
                        (hdr->policy == (uint32_t)pa.policy || hdr->t_next == 0);
    const int64_t t0 = hdr->t_next;
    const uint32_t parity = hdr->parity;

    if (active && hdr_ok) {
        const int b = chain / a.L, l = chain % a.L;
        const int N = a.N, L = a.L, T = a.T;
        const size_t row = (size_t)3 * N;
        uint32_t valid = 0u;
#pragma unroll
        for (int v = 0; v < V; ++v)
            if (lane * V + v < N) valid |= 1u << v;
        const bool has = valid != 0u;

        ChainState& cs = chains[chain];
        ChainRegs<V> cr;
        const uint32_t resident = lane_bits<V>(cs.bits, lane, N);
        cr.set_bits(resident);
        cr.count = (int)__reduce_add_sync(kFull, (uint32_t)__popc(resident));
        uint32_t aux[V];
        {
            Vec<V> x = load_vec<V>(val + (size_t)chain * N + lane * V, has);
#pragma unroll
            for (int v = 0; v < V; ++v) {
                cr.aT[v] = x.v[v];
                aux[v] = (has && lane * V + v < N) ? auxs[(size_t)chain * N + lane * V + v] : 0u;
            }
        }
        cr.hits = cr.misses = cr.pro = 0u;

        // running pointer to this lane's part of unit (b, t, l); p^S of rho(t, l)
        // at a fixed offset, the carry for the first token of layer 0
        const float* row0 = a.scores + ((size_t)b * T * L + l) * row;       // token 0 of the chain
        const float* carry_in = carry + ((size_t)parity * a.B + b) * N + lane * V;
        const size_t tok = (size_t)L * row;
        const ptrdiff_t s_off = l > 0 ? (ptrdiff_t)2 * N - (ptrdiff_t)row
                                      : (ptrdiff_t)(L - 1) * (ptrdiff_t)row - (ptrdiff_t)tok +
                                            (ptrdiff_t)2 * N;
        const bool want_s = POL == CRC_POLICY_SPATIO_LRU && a.R > 0;
        const bool rank_order = a.trace_topk != nullptr;

        // the rows pass through a ring in shared memory (ring_copy)
        constexpr int D = scan_ahead<V>();
        constexpr int ROWS = POL == CRC_POLICY_SPATIO_LRU ? 2 : 1;
        __shared__ __align__(16) float ring[kScanWarps][D][ROWS][32 * V];
        float (*mine)[ROWS][32 * V] = ring[(threadIdx.x >> 5) % kScanWarps];
        if (!has) {                              // slots past N read as 0
#pragma unroll
            for (int i = 0; i < D * ROWS; ++i)
#pragma unroll
                for (int v = 0; v < V; ++v) mine[i / ROWS][i % ROWS][lane * V + v] = 0.f;
        }
        const float* up = row0 + lane * V;
        auto load = [&](int t) {                 // t: the token `up` points at
            if (t < T && has) {
                ring_copy<V>(&mine[t % D][0][lane * V], up);
                if (want_s && t0 + t >= 1)
                    ring_copy<V>(&mine[t % D][ROWS - 1][lane * V],
                                 l == 0 && t == 0 ? carry_in : up + s_off);
            }
            ring_commit();
            up += tok;
        };
        // Top-K thresholds: lane j token t + j's; t's.  (A rank-order trace needs none.)
        // Taken within the step, or before it for Spatio-only, whose step holds more,
        // and for the widest network (40 streams x 600 tokens, Qwen3 shape, us,
        // before / within: LRU 385 / 380, LFU 412 / 404, LRFU 594 / 586, Spatio-only
        // 617 / 627; LFU, K = 32, 64 streams x 24 layers x 300 331 / 352).
        float theta = 0.f, th = 0.f;
        constexpr bool BEFORE = POL == CRC_POLICY_SPATIO_LRU || KP > 16;
        auto thresholds = [&](int t) {
            if (t + lane < T) theta = row_theta_k<KP>(row0 + (size_t)(t + lane) * tok, N, a.K);
            th = __shfl_sync(kFull, theta, 0);
        };
        auto step = [&](int t) {
            float pR[V], pS[V];
            ring_read<V>(&mine[t % D][0][lane * V], pR);
            ring_read<V>(&mine[t % D][ROWS - 1][lane * V], pS);
            if (!BEFORE && !rank_order && (t & 31) == 0) thresholds(t);
            Sel<V> s;
            const size_t unit = ((size_t)b * a.trace_T + a.trace_t0 + t) * L + l;
            if (rank_order)
                sel_from_bits<V>(
                    topk_ranked<V>(pR, valid, lane, a.K, a.trace_topk + unit * a.K), s);
            else
                sel_above<V, ALL_VALID>(pR, th, valid, s);
            policy_step<V, ALL_VALID, POL>(
                cr, aux, pR, pS, want_s && t0 + t >= 1, valid, lane, pa, (uint32_t)(t0 + t),
                s, [&](Sel<V>& x) { sel_ties<V>(pR, th, valid, lane, a.K, x); },
                a.trace_miss ? a.trace_miss + unit : nullptr,
                a.trace_pro ? a.trace_pro + unit : nullptr);
        };
#pragma unroll
        for (int t = 0; t < D - 1; ++t) load(t);
#pragma unroll 1
        for (int t = 0; t < T; ++t) {
            load(t + D - 1);
            if (BEFORE && !rank_order && (t & 31) == 0) thresholds(t);
            ring_wait<D - 1>();                  // token t's copies have landed
            step(t);
            th = __shfl_sync(kFull, theta, (t + 1) & 31);
        }

        // write back the chain
        const int NW = (N + 31) >> 5;
        for (int w = 0; w < NW; ++w) {
            const int e0 = lane * V;
            const uint32_t contrib = (has && (e0 >> 5) == w) ? (cr.bits(lane) << (e0 & 31)) : 0u;
            const uint32_t word = __reduce_or_sync(kFull, contrib);
            if (lane == 0) cs.bits[w] = word;
        }
        if (has) {
#pragma unroll
            for (int v = 0; v < V; ++v)
                if (lane * V + v < N) {
                    val[(size_t)chain * N + lane * V + v] = cr.aT[v];
                    auxs[(size_t)chain * N + lane * V + v] = aux[v];
                }
        }
        if (lane == 0) {
            cs.hits += cr.hits;
            cs.misses += cr.misses;
            cs.proactive += cr.pro;
        }
        // the last layer hands its final p^S to layer 0 of the next call
        if (l == L - 1 && has) {
            const float* src = row0 + lane * V + (size_t)(T - 1) * tok + 2 * N;
            float* dst = carry + ((size_t)(parity ^ 1u) * a.B + b) * N + lane * V;
#pragma unroll
            for (int v = 0; v < V; ++v)
                if (lane * V + v < N) dst[v] = src[v];
        }
    }

    // the last block to finish advances the token counter, flips the carry
    // slot and records the policy
    __syncthreads();
    if (threadIdx.x == 0) {
        if (!hdr_ok && blockIdx.x == 0) latch_error(&hdr->error, CRC_ESTATE);
        __threadfence();
        const uint32_t prev = atomicAdd(&hdr->done, 1u);
        if (prev == gridDim.x - 1) {
            __threadfence();
            if (hdr_ok) {
                hdr->t_next = t0 + a.T;
                hdr->parity = parity ^ 1u;
                hdr->policy = (uint32_t)pa.policy;
            }
            hdr->done = 0u;
            __threadfence();
        }
    }
}

}  // namespace crc
