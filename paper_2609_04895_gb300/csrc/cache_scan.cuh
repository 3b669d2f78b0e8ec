// Cache scan: one warp per (stream, layer) chain, sequential over tokens.
//
// Lane i owns experts [i*V, i*V + V).  Per access (Algorithm 2 of the paper
// with Algorithm 1 as its last step):
//   s^T  = p^R + p^T                                   (Sec. 3.2)
//   s^ST = s^T_{t-1} + p^S_{rho(t,l)}  (R > 0, t >= 1)  (Sec. 3.3)
//   refinement over A = Top_R(s^ST): skip residents, fill a free slot,
//   else replace the lowest resident when strictly higher; a candidate that
//   loses ends the refinement (every later one is no higher and the lowest
//   resident only rises, so it would lose too);
//   S = TopK(p^R); misses = |S \ C~|;
//   UpdateCache: demand-loaded experts fill free slots, then each further one
//   evicts the lowest-s^T resident outside S (the demand set's order does not
//   change the resulting set, since inserted experts are in S and protected).
// Reductions: the fp32 bit patterns of the (non-negative) scores are ordered
// like the scores, so a warp-wide extreme is a lane-local extreme and one
// redux.sync; the slot that holds it finds itself by comparing, and a count of
// the holders proves that there was exactly one.  Two holders (equal scores) go
// to the general forms, which settle every case by expert index with ballots.
//
// What bounds the step: the integer pipe (16 lanes a scheduler) when many
// chains share an SM, and for a few chains the latency of some 300 dependent
// instructions, a max/min redux.sync taking 23 cycles, an add 48.  So residency
// is held in floats and worked on by the FMA pipe.  Integer masks and selects
// with one reduction after another / this form, ms: Qwen3 shape, stand-alone scan
// of 64 streams x 1000 tokens, method 1.62 / 1.27, LRU 1.06 / 0.85, LFU 1.24 /
// 0.91, LRFU 1.39 / 1.31, Spatio-only 1.57 / 1.39; GPT-OSS shape (one expert a
// lane) 0.64 / 0.44, 0.34 / 0.32, 0.36 / 0.33, 0.43 / 0.43, 0.63 / 0.52; one
// stream through the fused kernel, 0.82 / 0.65 us a token.
#pragma once

#include "crc_device.cuh"

namespace crc {

struct ScanArgs {
    const float* scores;     // [B][T][L][3][N]
    uint8_t* state;          // state buffer base
    uint8_t* trace_topk;     // [B][T][L][K] or null
    uint8_t* trace_miss;     // [B][T][L] or null
    uint8_t* trace_pro;      // [B][T][L] or null
    uint32_t* trace_mid;     // [B][T][L][NW] cache after the refinement, or null
    uint32_t* trace_after;   // [B][T][L][NW] cache after UpdateCache, or null
    uint32_t* trace_sel;     // [B][T][L][NW] native Top-K set, or null
    int trace_T, trace_t0;   // trace arrays span trace_T tokens; this call starts at trace_t0
    int B, T, L, N, K, C, R;
};

// Keys: scores are non-negative, so their fp32 bit patterns are already
// ordered like the values; +1 keeps every real key above 0, which marks an
// empty slot.  Each lane keeps (key, slot) pairs sorted in policy order
// (key descending, equal keys by ascending slot = ascending expert index).
__device__ __forceinline__ uint32_t pkey(float x) { return __float_as_uint(x) + 1u; }
__device__ __forceinline__ uint32_t umin(uint32_t a, uint32_t b) { return a < b ? a : b; }
__device__ __forceinline__ uint32_t umax(uint32_t a, uint32_t b) { return a > b ? a : b; }

template <int V>
struct KeyList {
    uint32_t k[V];
    uint32_t s[V];
};

// Stable sort of a lane's V entries: odd-even transposition that swaps only
// strictly smaller keys forward, so equal keys keep their ascending slots.
template <int V>
__device__ __forceinline__ void presort(KeyList<V>& L) {
#pragma unroll
    for (int round = 0; round < V; ++round) {
#pragma unroll
        for (int j = round & 1; j + 1 < V; j += 2) {
            const bool sw = L.k[j + 1] > L.k[j];
            const uint32_t k0 = L.k[j], s0 = L.s[j];
            L.k[j] = sw ? L.k[j + 1] : k0;
            L.s[j] = sw ? L.s[j + 1] : s0;
            L.k[j + 1] = sw ? k0 : L.k[j + 1];
            L.s[j + 1] = sw ? s0 : L.s[j + 1];
        }
    }
}

template <int V>
struct Keys {
    uint32_t k[V];
};

// Removes the warp-wide first entry in policy order: the largest head key and,
// among lanes whose head has it, the lowest lane (lanes own ascending index
// ranges; a lane's head is its lowest index among equal keys).  Returns the
// owner lane (-1 when every list is empty); the owner receives the slot.
template <int V>
__device__ __forceinline__ int warp_pop_first(KeyList<V>& L, int lane, uint32_t& key,
                                              uint32_t& slot) {
    const uint32_t m = __reduce_max_sync(kFull, L.k[0]);
    key = m;
    const uint32_t b = __ballot_sync(kFull, m != 0u && L.k[0] == m);
    if (b == 0u) return -1;
    const int owner = __ffs(b) - 1;
    if (lane == owner) {
        slot = L.s[0];
#pragma unroll
        for (int j = 0; j + 1 < V; ++j) {
            L.k[j] = L.k[j + 1];
            L.s[j] = L.s[j + 1];
        }
        L.k[V - 1] = 0u;
    }
    return owner;
}

// The Top-K set of a row held by the warp (V keys a lane, 0 in invalid slots),
// as V bits a lane, equal keys by ascending index: K pops with one owner each.
template <int V>
__device__ __noinline__ uint32_t topk_ties(Keys<V> key, uint32_t valid, int lane, int K) {
    KeyList<V> P;
#pragma unroll
    for (int v = 0; v < V; ++v) {
        P.k[v] = ((valid >> v) & 1u) ? key.k[v] + 1u : 0u;
        P.s[v] = v;
    }
    presort<V>(P);
    uint32_t sel = 0u;
#pragma unroll 1
    for (int k = 0; k < K; ++k) {
        uint32_t kk, slot = 0u;
        const int owner = warp_pop_first<V>(P, lane, kk, slot);
        if (lane == owner) sel |= 1u << slot;
    }
    return sel;
}

// Last member in policy order among the slots flagged in `members`: smallest
// key and, among equal keys, the highest index.  Returns the owner lane (-1 if
// no member); the owner receives the slot.  Keys are >= 1, so a non-member
// counts as the largest key, 0xffffffff, which no real key reaches.
template <int V>
__device__ __forceinline__ int warp_last_member(const uint32_t (&k)[V], uint32_t members,
                                                int lane, uint32_t& key, uint32_t& slot) {
    uint32_t m[V];
#pragma unroll
    for (int v = 0; v < V; ++v) m[v] = ((members >> v) & 1u) ? k[v] : 0xffffffffu;
    uint32_t best = m[0];
#pragma unroll
    for (int v = 1; v < V; ++v) best = umin(best, m[v]);
    const uint32_t mn = __reduce_min_sync(kFull, best);
    key = mn;
    const uint32_t b = __ballot_sync(kFull, best == mn);
    if (mn == 0xffffffffu) return -1;
    const int owner = 31 - __clz(b);
    uint32_t bs = 0u;
#pragma unroll
    for (int v = 0; v < V; ++v) bs = m[v] == mn ? (uint32_t)v : bs;   // the highest such slot
    if (lane == owner) slot = bs;
    return owner;
}

template <int V>
struct Vec {
    float v[V];
};

// The stand-alone scans' rows pass through a ring in shared memory, filled
// with cp.async scan_ahead tokens ahead of use: a step takes less than a trip to
// L2 (480 cycles), let alone to DRAM, and a load into registers one step ahead
// is waited for at the step's end (N = 32, 40 streams x 600 tokens: 0.79 us a
// token for a chain's 144 instructions; 0.45 with the ring).  Every lane copies
// and reads its own V floats, so no barrier is needed.
template <int V>
constexpr int scan_ahead() { return V >= 4 ? 4 : 8; }

template <int V>
__device__ __forceinline__ void ring_copy(float* dst, const float* src) {
    const uint32_t at = smem_u32(dst);
    if constexpr (V == 8) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(at), "l"(src) : "memory");
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(at + 16u), "l"(src + 4)
                     : "memory");
    } else if constexpr (V == 4) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(at), "l"(src) : "memory");
    } else if constexpr (V == 2) {
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(at), "l"(src) : "memory");
    } else {
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(at), "l"(src) : "memory");
    }
}
__device__ __forceinline__ void ring_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int LEFT>
__device__ __forceinline__ void ring_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(LEFT) : "memory");
}
template <int V>
__device__ __forceinline__ void ring_read(const float* src, float (&x)[V]) {
    if constexpr (V >= 4) {
#pragma unroll
        for (int i = 0; i < V; i += 4) {
            const float4 f = *reinterpret_cast<const float4*>(src + i);
            x[i] = f.x;
            x[i + 1] = f.y;
            x[i + 2] = f.z;
            x[i + 3] = f.w;
        }
    } else if constexpr (V == 2) {
        const float2 f = *reinterpret_cast<const float2*>(src);
        x[0] = f.x;
        x[1] = f.y;
    } else {
        x[0] = *src;
    }
}

template <int V>
__device__ __forceinline__ Vec<V> load_vec(const float* p, bool ok) {
    Vec<V> r;
    if (!ok) {
#pragma unroll
        for (int i = 0; i < V; ++i) r.v[i] = 0.f;
        return r;
    }
    if constexpr (V == 4) {
        const float4 x = __ldg(reinterpret_cast<const float4*>(p));
        r.v[0] = x.x; r.v[1] = x.y; r.v[2] = x.z; r.v[3] = x.w;
    } else if constexpr (V == 2) {
        const float2 x = __ldg(reinterpret_cast<const float2*>(p));
        r.v[0] = x.x; r.v[1] = x.y;
    } else if constexpr (V == 8) {
        const float4 x = __ldg(reinterpret_cast<const float4*>(p));
        const float4 y = __ldg(reinterpret_cast<const float4*>(p) + 1);
        r.v[0] = x.x; r.v[1] = x.y; r.v[2] = x.z; r.v[3] = x.w;
        r.v[4] = y.x; r.v[5] = y.y; r.v[6] = y.z; r.v[7] = y.w;
    } else {
        r.v[0] = __ldg(p);
    }
    return r;
}

// ---------------------------------------------------------------------------
// The chain's step in fp32 arithmetic.  Residency is a 0 / 1 float per slot,
// so masking a score, counting and updating the cache are FMA-pipe operations;
// the integer pipe, whose 16 lanes a scheduler bound the scans when masks,
// counts and updates were selects and integer adds (5 warps x 365 instructions
// x 2 cycles a token for the Qwen3 shape), keeps the comparisons.
// ---------------------------------------------------------------------------
constexpr float kFar = 8.507059173023462e37f;   // 2^126; rows above it take the general forms

// 1.0 where the comparison holds, else 0.0
__device__ __forceinline__ float set_gt(float a, float b) {
    float r;
    asm("set.gt.f32.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float set_ge(float a, float b) {
    float r;
    asm("set.ge.f32.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float set_eq(float a, float b) {
    float r;
    asm("set.eq.f32.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}
// Largest / smallest over the warp of non-negative floats, on their bits (whose
// order is theirs; the compiler knows these reductions to be warp-uniform).
__device__ __forceinline__ float warp_max_f(float x) {
    return __uint_as_float(__reduce_max_sync(kFull, __float_as_uint(x)));
}
__device__ __forceinline__ float warp_min_f(float x) {
    return __uint_as_float(__reduce_min_sync(kFull, __float_as_uint(x)));
}
template <int V>
__device__ __forceinline__ float lane_min_f(const float (&x)[V]) {
    float r = x[0];
#pragma unroll
    for (int v = 1; v < V; ++v) r = fminf(r, x[v]);
    return r;
}
template <int V>
__device__ __forceinline__ float lane_max_f(const float (&x)[V]) {
    float r = x[0];
#pragma unroll
    for (int v = 1; v < V; ++v) r = fmaxf(r, x[v]);
    return r;
}
// Warp sum of lane values 2^23 + i, i a small whole number: the sum of the i.
constexpr float kCount0 = 8388608.f;
__device__ __forceinline__ uint32_t warp_count(float c) {
    return __reduce_add_sync(kFull, __float_as_uint(c)) - 0x60000000u;   // 32 * bits(2^23)
}

// Chain-local state held in registers across tokens.
template <int V>
struct ChainRegs {
    float out[V];        // 0 where this lane's expert is resident, else 1
    int count;           // |C| (warp-uniform)
    float aT[V];         // s^T of the previous token
    uint32_t hits, misses, pro;

    __device__ __forceinline__ uint32_t bits(int) const {    // the residency as V bits
        float b = kCount0 + (float)((1 << V) - 1);
#pragma unroll
        for (int v = 0; v < V; ++v) b = __fmaf_rn(out[v], -(float)(1 << v), b);
        return __float_as_uint(b) & ((1u << V) - 1u);
    }
    __device__ __forceinline__ void set_bits(uint32_t b) {
#pragma unroll
        for (int v = 0; v < V; ++v) out[v] = ((b >> v) & 1u) ? 0.f : 1.f;
    }
};

// Up to 32 experts, one a lane: the cache is one word, the same in every lane.
template <>
struct ChainRegs<1> {
    uint32_t cache;
    int count;
    float aT[1];
    uint32_t hits, misses, pro;

    __device__ __forceinline__ uint32_t bits(int lane) const { return (cache >> lane) & 1u; }
    __device__ __forceinline__ void set_bits(uint32_t b) {
        cache = __ballot_sync(kFull, b & 1u);
    }
};

// The native Top-K of an access: 0 / 1 per slot, or for one expert a lane the
// set as one word.
template <int V>
struct Sel {
    float s[V];
};
template <>
struct Sel<1> {
    uint32_t m;
};

// ---------------------------------------------------------------------------
// Thread-serial Top-K set of one score row (used for many tokens at once, one
// token per lane).  Sorting networks on fp32 values (max/min only) find the
// K-th largest value theta; a second pass in index order takes every value
// above theta and, among values equal to theta, the lowest indices -- exactly
// the first K under (score desc, index asc).
// ---------------------------------------------------------------------------
constexpr int pow2_at_least(int x) {
    int p = 1;
    while (p < x) p <<= 1;
    return p;
}

// Sort P values descending (P a power of two), fully unrolled: the bitonic
// network.
template <int P>
__device__ __forceinline__ void bitonic_sort_desc(float (&a)[P]) {
#pragma unroll
    for (int k = 2; k <= P; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
#pragma unroll
            for (int i = 0; i < P; ++i) {
                const int l = i ^ j;
                if (l > i) {
                    const float hi = fmaxf(a[i], a[l]), lo = fminf(a[i], a[l]);
                    if ((i & k) == 0) {
                        a[i] = hi;
                        a[l] = lo;
                    } else {
                        a[i] = lo;
                        a[l] = hi;
                    }
                }
            }
        }
    }
}

// The same with Batcher's odd-even merge sort, which sorts P = 4 with 5
// compare-exchanges and P = 8 with 19 (the bitonic network takes 6 and 24).
// Stage p merges sorted runs of p into runs of 2p; within it, the
// compare-exchanges at distance k join elements of the same run of 2p.  Used
// up to P = 8; beyond that the compiler no longer resolves every index.
template <int P>
__device__ __forceinline__ void sort_desc(float (&a)[P]) {
    if constexpr (P > 8) {
        bitonic_sort_desc<P>(a);
    } else {
#pragma unroll
        for (int p = 1; p < P; p <<= 1) {
#pragma unroll
            for (int k = p; k >= 1; k >>= 1) {
#pragma unroll
                for (int j = k % p; j + k < P; j += 2 * k) {
#pragma unroll
                    for (int i = 0; i < k; ++i) {
                        const int x = i + j, y = i + j + k;
                        if (y < P && x / (2 * p) == y / (2 * p)) {
                            const float hi = fmaxf(a[x], a[y]), lo = fminf(a[x], a[y]);
                            a[x] = hi;
                            a[y] = lo;
                        }
                    }
                }
            }
        }
    }
}

// run <- the P largest of (run, b), both sorted descending; result descending.
template <int P>
__device__ __forceinline__ void merge_top_desc(float (&run)[P], const float (&b)[P]) {
#pragma unroll
    for (int i = 0; i < P; ++i) run[i] = fmaxf(run[i], b[P - 1 - i]);   // bitonic
#pragma unroll
    for (int j = P >> 1; j > 0; j >>= 1) {
#pragma unroll
        for (int i = 0; i < P; ++i) {
            const int l = i ^ j;
            if (l > i) {
                const float hi = fmaxf(run[i], run[l]), lo = fminf(run[i], run[l]);
                run[i] = hi;
                run[l] = lo;
            }
        }
    }
}

// Running top-KP values (descending) of a stream of non-negative scores fed 16
// at a time; theta(K) is then the K-th largest score and need(K) how many of
// the scores equal to theta belong to the Top-K set (the lowest indices).
template <int KP>
struct TopKAcc {
    float run[KP];
    __device__ __forceinline__ void init() {
#pragma unroll
        for (int i = 0; i < KP; ++i) run[i] = -1.0f;   // below every score
    }
    __device__ __forceinline__ void add16(const float* x) {
        constexpr int G = KP < 16 ? KP : 16;
#pragma unroll
        for (int g = 0; g < 16; g += G) {
            float b[KP];
#pragma unroll
            for (int i = 0; i < KP; ++i) b[i] = (i < G) ? x[g + i] : -1.0f;
            sort_desc<KP>(b);
            merge_top_desc<KP>(run, b);
        }
    }
    __device__ __forceinline__ float theta(int K) const {
        float th = run[0];
#pragma unroll
        for (int i = 0; i < KP; ++i)
            if (i == K - 1) th = run[i];
        return th;
    }
    __device__ __forceinline__ int need(int K, float th) const {
        int gt = 0;
#pragma unroll
        for (int i = 0; i < KP; ++i)
            if (i < K && run[i] > th) ++gt;
        return K - gt;
    }
};

// Threshold pass over 4 consecutive scores: take everything above theta and the
// first `need` scores equal to theta; returns the 4 bits.
__device__ __forceinline__ uint32_t take4(float4 f, float th, int& need) {
    const float v[4] = {f.x, f.y, f.z, f.w};
    uint32_t w = 0u;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const bool eq = v[u] == th;
        const bool take = (v[u] > th) || (eq && need > 0);
        need -= eq ? 1 : 0;
        w |= take ? (1u << u) : 0u;
    }
    return w;
}

// K-th largest of row[0..N) (N % 16 == 0, 1 <= K <= min(N, 32), values >= 0):
// the threshold of its Top-K set, which is every score at or above it unless
// more than K are.
template <int KP>
__device__ __forceinline__ float row_theta_k(const float* row, int N, int K) {
    TopKAcc<KP> acc;
    acc.init();
    for (int c = 0; c < N; c += 16) {
        float x[16];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float4 f = __ldg(reinterpret_cast<const float4*>(row + c) + q);
            x[4 * q] = f.x;
            x[4 * q + 1] = f.y;
            x[4 * q + 2] = f.z;
            x[4 * q + 3] = f.w;
        }
        acc.add16(x);
    }
    return acc.theta(K);
}

// Algorithm 2's pre-access refinement of the chain's cache with priorities
// a[e] + pS[e] (s^ST for the method, s^S for the Spatio-only ablation): the
// candidates A = Top_R of all experts in descending order, each skipped when
// resident, loaded into a free slot, or swapped for the lowest resident when
// strictly higher.  Returns the proactive loads.
//
// Only the non-resident members of A can change the cache, so they are taken
// one at a time in order -- the best remaining non-resident c -- and c is a
// member of A = Top_R exactly when fewer than R experts precede it in the
// order (its rank).  The first rank test is also the one that leaves the cache
// alone when the R first experts are all resident.  An original resident that
// a candidate evicted is never taken as a candidate itself: in the literal
// loop it would meet a cache whose lowest member is no lower than it and lose
// the strict test, ending the pass exactly as the rank test or the strict
// test ends it here.
//
// The general form, for ties (keys: score bits, 0 in invalid slots).  A function of its own, so the scans' loops stay short.
// Returns the cache (V bits) | its count << 8 | the proactive loads << 20.
template <int V>
__device__ __noinline__ uint32_t refine_general(Keys<V> key, uint32_t cache, int count,
                                                uint32_t valid, int lane, int C, int R) {
    uint32_t kS[V];                            // the keys + 1, 0 in invalid slots
#pragma unroll
    for (int v = 0; v < V; ++v) kS[v] = ((valid >> v) & 1u) ? key.k[v] + 1u : 0u;
    uint32_t left = valid & ~cache;            // non-residents not yet taken
    int pro = 0;
#pragma unroll 1
    for (int j = 0; j < R; ++j) {
        // the best remaining non-resident c: largest key, then lowest index
        uint32_t m[V];
#pragma unroll
        for (int v = 0; v < V; ++v) m[v] = ((left >> v) & 1u) ? kS[v] : 0u;
        uint32_t best = m[0];
#pragma unroll
        for (int v = 1; v < V; ++v) best = umax(best, m[v]);
        const uint32_t mx = __reduce_max_sync(kFull, best);
        if (mx == 0u) break;                   // no non-resident left
        const int owner = __ffs(__ballot_sync(kFull, best == mx)) - 1;
        uint32_t cs = 0u;
#pragma unroll
        for (int v = V - 1; v >= 0; --v) cs = m[v] == mx ? (uint32_t)v : cs;   // lowest slot
        const uint32_t c_slot = __shfl_sync(kFull, cs, owner);
        // rank of c: experts with higher keys, and with equal keys at lower indices
        uint32_t before = 0u;
#pragma unroll
        for (int v = 0; v < V; ++v)
            before += (kS[v] > mx ||
                       (kS[v] == mx && (lane < owner || (lane == owner && (uint32_t)v < c_slot))))
                          ? 1u : 0u;
        if ((int)__reduce_add_sync(kFull, before) >= R) break;   // nor is any later one in A
        const uint32_t cbit = (lane == owner) ? (1u << cs) : 0u;
        left &= ~cbit;
        if (count < C) {                       // free slot: proactive load
            cache |= cbit;
            ++count;
            ++pro;
            continue;
        }
        uint32_t kv, vslot = 0u;
        const int vo = warp_last_member<V>(kS, cache, lane, kv, vslot);
        if (mx <= kv) break;                   // later candidates are no higher
        const uint32_t vbit = (lane == vo) ? (1u << vslot) : 0u;
        cache = (cache & ~vbit) | cbit;        // strictly higher: replace the lowest resident
        ++pro;
    }
    return cache | ((uint32_t)count << 8) | ((uint32_t)pro << 20);
}

// This lane's share of two counts over the warp: the demand misses of the
// slots s (at most K <= 32) and, times 64, the members of s.
template <int V>
__device__ __forceinline__ float miss_count(const ChainRegs<V>& cr, const Sel<V>& sel) {
    float miss = 0.f, all = 0.f;
#pragma unroll
    for (int v = 0; v < V; ++v) {
        miss = __fmaf_rn(sel.s[v], cr.out[v], miss);
        all = __fadd_rn(all, sel.s[v]);
    }
    return __fmaf_rn(all, 64.f, miss);
}

// The refinement: a round takes the best non-resident's score and the lowest
// resident's in two independent reductions, then one count that carries both
// c's rank and the demand misses of the native Top-K s against the cache as it
// stands, so the round that ends the pass has also counted them.  A load or a
// swap is made by the slots that hold the two scores, after a count has shown
// that each has one holder, c's among all experts and the lowest's among the
// residents; otherwise refine_general takes the pass on from the cache as it
// is.
// *counts receives the demand misses and, above bit 6, the members of s.
template <int V, bool ALL_VALID>
__device__ __forceinline__ int scan_refine(ChainRegs<V>& cr, const float (&pS)[V], uint32_t valid,
                                           int lane, int C, int R, const Sel<V>& s,
                                           uint32_t* counts) {
    float k[V];
#pragma unroll
    for (int v = 0; v < V; ++v) {
        k[v] = __fadd_rn(cr.aT[v], pS[v]);
        if (!ALL_VALID && !((valid >> v) & 1u)) k[v] = 0.f;
    }
    int pro = 0;
    bool general = false;
#pragma unroll 1
    while (true) {
        const bool full = cr.count == C;
        float x[V], y[V];
#pragma unroll
        for (int v = 0; v < V; ++v) {
            x[v] = __fmul_rn(k[v], cr.out[v]);                 // invalid slots: 0
            y[v] = __fmaf_rn(cr.out[v], kFar, k[v]);
        }
        const float mx = warp_max_f(lane_max_f<V>(x));
        const float mn = warp_min_f(lane_min_f<V>(y));
        float gt = kCount0;
#pragma unroll
        for (int v = 0; v < V; ++v) gt = __fadd_rn(gt, set_gt(k[v], mx));
        const uint32_t tot = warp_count(__fmaf_rn(miss_count<V>(cr, s), 1024.f, gt));
        *counts = tot >> 10;
        // not among the top R, or no higher than the lowest resident of a full
        // cache: neither is any later candidate
        if ((int)(tot & 1023u) >= R || (full && __float_as_uint(mx) <= __float_as_uint(mn))) break;
        const float lowest = full ? mn : -1.f;                 // who leaves; nobody
        float h = kCount0, in[V], go[V];
#pragma unroll
        for (int v = 0; v < V; ++v) {
            in[v] = set_eq(k[v], mx);
            go[v] = set_eq(y[v], lowest);
            h = __fadd_rn(h, in[v]);
            h = __fmaf_rn(go[v], 1024.f, h);
        }
        general = warp_count(h) != (full ? 1025u : 1u) || mn >= kFar || mx == 0.f;
        if (general) break;
#pragma unroll
        for (int v = 0; v < V; ++v)
            cr.out[v] = __fadd_rn(__fsub_rn(cr.out[v], in[v]), go[v]);
        cr.count += full ? 0 : 1;
        ++pro;
    }
    if (general) {
        Keys<V> key;
#pragma unroll
        for (int v = 0; v < V; ++v) key.k[v] = __float_as_uint(k[v]);
        const uint32_t r = refine_general<V>(key, cr.bits(lane), cr.count, valid, lane, C, R);
        cr.set_bits(r & 0xffu);
        cr.count = (int)((r >> 8) & 0xfffu);
        pro += (int)(r >> 20);
        *counts = warp_count(__fadd_rn(miss_count<V>(cr, s), kCount0));
    }
    return pro;
}

// The members (V bits) left after the n with the smallest keys, ties to the
// highest index, are taken out one at a time.
template <int V>
__device__ __noinline__ uint32_t evict_general(Keys<V> key, uint32_t set, int n, int lane) {
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
        uint32_t kv, vslot = 0u;
        const int vo = warp_last_member<V>(key.k, set, lane, kv, vslot);
        if (lane == vo) set &= ~(1u << vslot);
    }
    return set;
}

// UpdateCache on a cache that overflows by n: of the residents outside S the n
// with the smallest keys (ties to the highest index) leave, and S comes in;
// `stay` of the former remain (their number is known: C - K).  Each round takes
// every slot that holds the minimum; when a count then shows that equal keys
// took more than n, the members are taken one at a time instead.  Ties are
// rare among sums of probabilities (KeyTies::kRare); keys may also be known to
// be distinct (kNone), or tie often (kOften: each round takes the highest
// index among the holders of the minimum, one more reduction).
enum class KeyTies { kNone, kRare, kOften };
template <int V, KeyTies TIES>
__device__ __forceinline__ void update_cache(ChainRegs<V>& cr, const float (&key)[V],
                                             const Sel<V>& sel, int n, int stay, int lane) {
    float y[V];
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const float not_in = __fadd_rn(cr.out[v], __fmaf_rn(-cr.out[v], sel.s[v], sel.s[v]));
        y[v] = __fmaf_rn(not_in, kFar, key[v]);
    }
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
        const float mn = warp_min_f(lane_min_f<V>(y));
        if constexpr (TIES == KeyTies::kOften) {
            uint32_t at = 0u;                  // 1 + the highest index here that holds it
#pragma unroll
            for (int v = 0; v < V; ++v) at = y[v] == mn ? (uint32_t)(lane * V + v + 1) : at;
            const uint32_t last = __reduce_max_sync(kFull, at);
#pragma unroll
            for (int v = 0; v < V; ++v)
                y[v] = (uint32_t)(lane * V + v + 1) == last ? kFar : y[v];
        } else {
#pragma unroll
            for (int v = 0; v < V; ++v) y[v] = __fmaf_rn(set_eq(y[v], mn), kFar, y[v]);
        }
    }
    float gone[V], c = kCount0;
#pragma unroll
    for (int v = 0; v < V; ++v) {
        gone[v] = set_ge(y[v], kFar);
        c = __fadd_rn(c, gone[v]);
    }
    if (TIES == KeyTies::kRare && warp_count(c) != (uint32_t)(32 * V - stay)) {
        Keys<V> all;
        uint32_t set = 0u;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            all.k[v] = __float_as_uint(key[v]);
            set |= (cr.out[v] == 0.f && sel.s[v] == 0.f) ? 1u << v : 0u;
        }
        set = evict_general<V>(all, set, n, lane);
#pragma unroll
        for (int v = 0; v < V; ++v) gone[v] = ((set >> v) & 1u) ? 0.f : 1.f;
    }
#pragma unroll
    for (int v = 0; v < V; ++v) cr.out[v] = __fmaf_rn(-sel.s[v], gone[v], gone[v]);
}

// The set of which a lane holds the V low bits of `bits`.
template <int V>
__device__ __forceinline__ void sel_from_bits(uint32_t bits, Sel<V>& sel) {
    if constexpr (V == 1) {
        sel.m = __ballot_sync(kFull, bits & 1u);
    } else {
#pragma unroll
        for (int v = 0; v < V; ++v) sel.s[v] = (bits & (1u << v)) ? 1.f : 0.f;
    }
}

// ---------------------------------------------------------------------------
// One expert a lane (N <= 32): sets are words and counts are popcounts of
// them, ties a choice of bit, so there is no general form to fall back to.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int refine_mask(ChainRegs<1>& cr, float pS, uint32_t valid, int lane,
                                           int C, int R) {
    const uint32_t bit = 1u << lane;
    const uint32_t key = valid ? __float_as_uint(__fadd_rn(cr.aT[0], pS)) + 1u : 0u;
    uint32_t left = __ballot_sync(kFull, valid != 0u) & ~cr.cache;   // not taken yet
    int pro = 0;
#pragma unroll 1
    for (int j = 0; j < R; ++j) {
        // the best remaining non-resident (ties: the lowest index), and the
        // lowest resident (ties: the highest)
        const uint32_t x = (left & bit) ? key : 0u;
        const uint32_t y = (cr.cache & bit) ? key : 0xffffffffu;
        const uint32_t mx = __reduce_max_sync(kFull, x);
        const uint32_t mn = __reduce_min_sync(kFull, y);
        const uint32_t c = __ballot_sync(kFull, x == mx) & left;
        const uint32_t cbit = c & (0u - c);
        const uint32_t ahead = __ballot_sync(kFull, key > mx) |
                               (__ballot_sync(kFull, key == mx) & (cbit - 1u));
        if (left == 0u || __popc(ahead) >= R) break;
        left &= ~cbit;
        if (cr.count < C) {
            cr.cache |= cbit;
            ++cr.count;
        } else {
            if (mx <= mn) break;
            const uint32_t v = __ballot_sync(kFull, y == mn) & cr.cache;
            cr.cache = (cr.cache & ~(0x80000000u >> __clz(v))) | cbit;
        }
        ++pro;
    }
    return pro;
}

// UpdateCache: of the residents outside `sel` the n with the smallest keys
// leave (ties: the highest index), then `sel` is resident.
__device__ __forceinline__ void update_mask(ChainRegs<1>& cr, uint32_t key, uint32_t sel, int n,
                                            int lane) {
    uint32_t w = cr.cache & ~sel;
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
        const uint32_t y = ((w >> lane) & 1u) ? key : 0xffffffffu;
        const uint32_t mn = __reduce_min_sync(kFull, y);
        const uint32_t v = __ballot_sync(kFull, y == mn) & w;
        w &= ~(0x80000000u >> __clz(v));
    }
    cr.cache = w | sel;
}

// Refinement, access and UpdateCache of one access, given s^T = p^R + p^T,
// the Spatio prediction of the predecessor and the native Top-K as slots s (0
// or 1), or as a word.  The counts show whether s has K members; if it has more (it was
// taken by its threshold and scores tie there), exact_set(s) puts it right.
// Updates the chain registers; returns the number of proactive loads and
// writes the demand misses to *n_miss.  after_refine() is called between the
// two phases.
template <int V, bool ALL_VALID, class X, class F>
__device__ __forceinline__ int scan_apply(ChainRegs<V>& cr, const float (&sT)[V],
                                          const float (&pS)[V], bool refine, uint32_t valid,
                                          int lane, int K, int C, int R, Sel<V>& s,
                                          int* n_miss, X exact_set, F after_refine) {
    int pro = 0, nD;
    if constexpr (V == 1) {
        if (refine) pro = refine_mask(cr, pS[0], valid, lane, C, R);
        after_refine();
        if (__popc(s.m) != K) exact_set(s);
        nD = __popc(s.m & ~cr.cache);
        const int over = cr.count + nD - C;
        update_mask(cr, __float_as_uint(sT[0]), s.m, over, lane);
        cr.count = over > 0 ? C : cr.count + nD;
    } else {
        uint32_t counts;
        if (refine)
            pro = scan_refine<V, ALL_VALID>(cr, pS, valid, lane, C, R, s, &counts);
        else
            counts = warp_count(__fadd_rn(miss_count<V>(cr, s), kCount0));
        after_refine();
        if ((counts >> 6) != (uint32_t)K) {
            exact_set(s);
            counts = warp_count(__fadd_rn(miss_count<V>(cr, s), kCount0));
        }
        nD = (int)(counts & 63u);

        // demand misses and UpdateCache (Algorithm 1)
        const int over = cr.count + nD - C;
        if (over > 0) {
            update_cache<V, KeyTies::kRare>(cr, sT, s, over, C - K, lane);
            cr.count = C;
        } else if (nD > 0) {
#pragma unroll
            for (int v = 0; v < V; ++v) cr.out[v] = __fmaf_rn(-s.s[v], cr.out[v], cr.out[v]);
            cr.count += nD;
        }
    }
#pragma unroll
    for (int v = 0; v < V; ++v) cr.aT[v] = sT[v];
    cr.hits += (uint32_t)(K - nD);
    cr.misses += (uint32_t)nD;
    cr.pro += (uint32_t)pro;
    *n_miss = nD;
    return pro;
}

// The slots at or above the Top-K threshold of the row p.
template <int V, bool ALL_VALID>
__device__ __forceinline__ void sel_above(const float (&p)[V], float theta, uint32_t valid,
                                          Sel<V>& sel) {
    if constexpr (V == 1) {
        sel.m = __ballot_sync(kFull, valid != 0u && p[0] >= theta);
    } else {
#pragma unroll
        for (int v = 0; v < V; ++v)
            sel.s[v] = (ALL_VALID || ((valid >> v) & 1u)) ? set_ge(p[v], theta) : 0.f;
    }
}
// The Top-K set (V bits a lane) of a row whose threshold th has more equals than
// the set takes: every score above it and, of the scores equal to it, the lowest
// indices.  A lane's numbers of the two are added up over the warp, and over the
// lanes before it, by ballots of their bits.  (K pops with one owner each,
// topk_ties, cost a tied row more than the rest of its step: LRU, N = 128, one
// stream x 24 layers x 300 tokens of tied rows, K = 32 873 us by pops, 235 by the
// threshold.)  Rows that no threshold settles (NaN) are left to them.
template <int V>
__device__ __noinline__ uint32_t topk_at(Vec<V> p, float th, uint32_t valid, int lane, int K) {
    uint32_t above = 0u, equal = 0u;
#pragma unroll
    for (int v = 0; v < V; ++v) {
        above |= p.v[v] > th ? 1u << v : 0u;
        equal |= p.v[v] == th ? 1u << v : 0u;
    }
    above &= valid;
    equal &= valid;
    const uint32_t a = __popc(above), e = __popc(equal);
    int n_above = 0, n_equal = 0, before = 0;
#pragma unroll
    for (int b = 0; (1 << b) <= V; ++b) {
        const uint32_t wa = __ballot_sync(kFull, (a >> b) & 1u);
        const uint32_t we = __ballot_sync(kFull, (e >> b) & 1u);
        n_above += __popc(wa) << b;
        n_equal += __popc(we) << b;
        before += __popc(we & ((1u << lane) - 1u)) << b;
    }
    const int need = K - n_above;
    if (need < 0 || need > n_equal) {
        Keys<V> key;
#pragma unroll
        for (int v = 0; v < V; ++v) key.k[v] = __float_as_uint(p.v[v]);
        return topk_ties<V>(key, valid, lane, K);
    }
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const bool eq = (equal >> v) & 1u;
        if (eq && before < need) above |= 1u << v;
        before += eq ? 1 : 0;
    }
    return above;
}
template <int V>
__device__ __forceinline__ void sel_ties(const float (&p)[V], float th, uint32_t valid, int lane,
                                         int K, Sel<V>& sel) {
    Vec<V> row;
#pragma unroll
    for (int v = 0; v < V; ++v) row.v[v] = p[v];
    sel_from_bits<V>(topk_at<V>(row, th, valid, lane, K), sel);
}
// This lane's V bits of the set.
template <int V>
__device__ __forceinline__ uint32_t sel_bits(const Sel<V>& sel, int lane) {
    if constexpr (V == 1) {
        return (sel.m >> lane) & 1u;
    } else {
        float b = kCount0;
#pragma unroll
        for (int v = 0; v < V; ++v) b = __fmaf_rn(sel.s[v], (float)(1 << v), b);
        return __float_as_uint(b) & ((1u << V) - 1u);
    }
}

// This lane's V bits of a set as the set's NW bitmask words at dst (4-byte
// aligned): the warp's bits are gathered to whole bytes (one ballot for V = 1;
// log2(8 / V) shuffles otherwise) and stored bytewise, 4 NW bytes in one
// store.  (One redux.or and one store a word took four of each for N = 128.)
template <int V>
__device__ __forceinline__ void store_cache_words(uint32_t bits, int lane, int N, uint32_t* dst) {
    const int NW = (N + 31) >> 5;
    if constexpr (V == 1) {
        const uint32_t word = __ballot_sync(kFull, bits & 1u);
        if (lane == 0) dst[0] = word;
    } else {
#pragma unroll
        for (int o = 1; o * V < 8; o <<= 1)
            bits |= __shfl_down_sync(kFull, bits, o) << (o * V);
        const int byte = lane * V / 8;
        if (lane % (8 / V) == 0 && byte < 4 * NW)
            reinterpret_cast<uint8_t*>(dst)[byte] = (uint8_t)bits;
    }
}

// The native Top-K in rank order, for a trace that wants it: returns the set.
template <int V>
__device__ __forceinline__ uint32_t topk_ranked(const float (&pR)[V], uint32_t valid, int lane,
                                                int K, uint8_t* topk_out) {
    KeyList<V> P;
#pragma unroll
    for (int v = 0; v < V; ++v) {
        P.k[v] = ((valid >> v) & 1u) ? pkey(pR[v]) : 0u;
        P.s[v] = v;
    }
    presort<V>(P);
    uint32_t sel = 0u;
    int mine = 0;
    for (int k = 0; k < K; ++k) {
        uint32_t kk, slot = 0u;
        const int owner = warp_pop_first<V>(P, lane, kk, slot);
        if (lane == owner) sel |= 1u << slot;
        const int e = __shfl_sync(kFull, lane * V + (int)slot, owner);
        if (lane == k) mine = e;
    }
    if (lane < K) topk_out[lane] = (uint8_t)mine;
    return sel;
}

// Bits of this lane's experts from the chain's bitmask words.
template <int V>
__device__ __forceinline__ uint32_t lane_bits(const uint32_t* words, int lane, int N) {
    const int e0 = lane * V;
    if (e0 >= N) return 0u;
    return (words[e0 >> 5] >> (e0 & 31)) & ((1u << V) - 1u);
}

// Warps (chains) per block of the stand-alone scans.  The scans are
// issue-bound with every chain resident at once, so their time is that of the
// most loaded SM: one-warp blocks spread the B*L chains within one warp per SM
// of even (3,072 chains over 152 SMs: 20 or 21 warps each, where blocks of
// four put 24 on some SMs and 20 on the rest).
constexpr int kScanWarps = 1;

// TRACED: compiled with the trace writes (any trace array given); the
// untraced kernel carries none of their code.
template <int V, bool ALL_VALID, int KP, bool TRACED>
__global__ void __launch_bounds__(32 * kScanWarps, (V >= 8 ? 12 : 24) / kScanWarps)
    cache_scan_kernel(ScanArgs a) {
    StateHeader* hdr = reinterpret_cast<StateHeader*>(a.state);
    const StateLayout lay = state_layout(a.B, a.L, a.N);
    ChainState* chains = reinterpret_cast<ChainState*>(a.state + lay.chains);
    float* retention = reinterpret_cast<float*>(a.state + lay.retention);
    float* carry = reinterpret_cast<float*>(a.state + lay.carry);

    const int lane = threadIdx.x & 31;
    const int chain = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const bool active = chain < a.B * a.L;

    const bool hdr_ok = hdr->magic == kStateMagic && hdr->L == a.L && hdr->N == a.N &&
                        hdr->K == a.K && hdr->C == a.C && hdr->R == a.R && hdr->B == a.B &&
                        hdr->policy == 0u;
    const int64_t t0 = hdr->t_next;
    const uint32_t parity = hdr->parity;

    uint32_t* err = &hdr->error;
    (void)err;                                  // read only by the checking build's bounds checks
    if (active && hdr_ok && CRC_IN_BOUNDS(a.trace_t0 >= 0 && a.trace_t0 + a.T <= a.trace_T, err)) {
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
        {
            Vec<V> x = load_vec<V>(retention + (size_t)chain * N + lane * V, has);
#pragma unroll
            for (int v = 0; v < V; ++v) cr.aT[v] = x.v[v];
        }
        cr.hits = cr.misses = cr.pro = 0u;

        // debug builds: the unit a pointer is formed for lies inside scores [B][T][L]
        auto unit_ok = [&](int t, int ll) {
            return CRC_IN_BOUNDS(b < a.B && t >= 0 && t < T && ll >= 0 && ll < L, err);
        };
        // running pointer to this lane's part of unit (b, t, l); p^S of rho(t, l)
        // sits at a fixed offset from it: unit (t, l-1), or (t-1, L-1) for l = 0,
        // whose first token takes the carry
        const float* row0 = a.scores + ((size_t)b * T * L + l) * row;       // token 0 of the chain
        const float* carry_in = carry + ((size_t)parity * a.B + b) * N + lane * V;
        const size_t tok = (size_t)L * row;
        const ptrdiff_t s_off = l > 0 ? (ptrdiff_t)2 * N - (ptrdiff_t)row
                                      : (ptrdiff_t)(L - 1) * (ptrdiff_t)row - (ptrdiff_t)tok +
                                            (ptrdiff_t)2 * N;
        const bool want_s = a.R > 0;
        const bool rank_order = TRACED && a.trace_topk != nullptr;

        constexpr int D = scan_ahead<V>();
        __shared__ __align__(16) float ring[kScanWarps][D][3][32 * V];
        float (*mine)[3][32 * V] = ring[(threadIdx.x >> 5) % kScanWarps];
        if (!has) {                              // slots past N read as 0
#pragma unroll
            for (int i = 0; i < D * 3; ++i)
#pragma unroll
                for (int v = 0; v < V; ++v) mine[i / 3][i % 3][lane * V + v] = 0.f;
        }
        const float* up = row0 + lane * V;
        auto load = [&](int t) {                 // t: the token `up` points at
            if (t < T && has && unit_ok(t, l)) {
                float (*to)[32 * V] = mine[t % D];
                const bool first = l == 0 && t == 0;
                ring_copy<V>(&to[0][lane * V], up);
                ring_copy<V>(&to[1][lane * V], up + N);
                if (want_s && t0 + t >= 1 &&
                    (first || unit_ok(l > 0 ? t : t - 1, l > 0 ? l - 1 : L - 1)))
                    ring_copy<V>(&to[2][lane * V], first ? carry_in : up + s_off);
            }
            ring_commit();
            up += tok;
        };
        // The Top-K thresholds do not depend on the cache: lane j takes that of
        // token t + j for t a multiple of 32; th is the current token's.  A
        // rank-order trace takes the whole order instead and needs none (one
        // token, N = 128, K = 32, 64 streams x 24 layers: 24.6 us with the
        // thresholds, 9.5 without).  They are taken within the step, or before it
        // for the widest network, whose registers weigh on it (us, before / within:
        // K = 8, 40 streams x 600 tokens, Qwen3 shape, 598 / 588; N = 128, 64 streams
        // x 24 layers x 300, K = 16 320 / 307, K = 32 405 / 451).
        float theta = 0.f, th = 0.f;
        constexpr bool BEFORE = KP > 16;
        auto thresholds = [&](int t) {
            if (t + lane < T && unit_ok(t + lane, l))
                theta = row_theta_k<KP>(row0 + (size_t)(t + lane) * tok, N, a.K);
            th = __shfl_sync(kFull, theta, 0);
        };
        auto step = [&](int t) {
            float pR[V], pT[V], pS[V];
            float (*from)[32 * V] = mine[t % D];
            ring_read<V>(&from[0][lane * V], pR);
            ring_read<V>(&from[1][lane * V], pT);
            ring_read<V>(&from[2][lane * V], pS);
            if (!BEFORE && !rank_order && (t & 31) == 0) thresholds(t);
            Sel<V> s;
            float sT[V];
            if (!rank_order) sel_above<V, ALL_VALID>(pR, th, valid, s);
            const size_t unit = ((size_t)b * a.trace_T + a.trace_t0 + t) * L + l;
            const size_t NWs = (size_t)((N + 31) >> 5);
            if (rank_order)
                sel_from_bits<V>(
                    topk_ranked<V>(pR, valid, lane, a.K, a.trace_topk + unit * a.K), s);
#pragma unroll
            for (int v = 0; v < V; ++v) sT[v] = __fadd_rn(pR[v], pT[v]);
            int nD;
            const int pro = scan_apply<V, ALL_VALID>(
                cr, sT, pS, want_s && t0 + t >= 1, valid, lane, a.K, a.C, a.R, s, &nD,
                [&](Sel<V>& x) { sel_ties<V>(pR, th, valid, lane, a.K, x); },
                [&] {
                    if (TRACED && a.trace_mid)
                        store_cache_words<V>(cr.bits(lane), lane, N, a.trace_mid + unit * NWs);
                });
            if constexpr (TRACED) {
                if (a.trace_after)
                    store_cache_words<V>(cr.bits(lane), lane, N, a.trace_after + unit * NWs);
                if (a.trace_sel)
                    store_cache_words<V>(sel_bits<V>(s, lane), lane, N, a.trace_sel + unit * NWs);
                if (lane == 0) {
                    if (a.trace_miss) a.trace_miss[unit] = (uint8_t)nD;
                    if (a.trace_pro) a.trace_pro[unit] = (uint8_t)pro;
                }
            }
            // debug builds: every expert the step made resident lies in this
            // lane's range and the cache holds at most C experts
            (void)CRC_IN_BOUNDS((cr.bits(lane) & ~valid) == 0u && cr.count <= a.C, err);
        };
#pragma unroll
        for (int t = 0; t < D - 1; ++t) load(t);
        // (One copy of the step in the loop: two, with registers in place of the
        // ring, ran a lone chain 13 % slower for the longer code.)
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
        if (has && CRC_IN_BOUNDS(chain < a.B * a.L, err)) {
#pragma unroll
            for (int v = 0; v < V; ++v)
                if (lane * V + v < N) retention[(size_t)chain * N + lane * V + v] = cr.aT[v];
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

    // the last block to finish advances the token counter and flips the carry slot
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
            }
            hdr->done = 0u;
            __threadfence();
        }
    }
}

}  // namespace crc
