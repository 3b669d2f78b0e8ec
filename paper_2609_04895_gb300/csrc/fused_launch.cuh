// Host side of the fused route-and-cache kernel: tile plan, workspace layout,
// tensor maps and the cooperative launch (all CTAs resident at once, which the
// kernel's producer / consumer waits rely on).
#pragma once

#include <algorithm>
#include <cstdlib>

#include "crc_internal.h"
#include "fused.cuh"

namespace crc {

inline bool plain_cluster_launch() {
    static const bool on = [] {
        const char* v = std::getenv("CRC_PLAIN_CLUSTER_LAUNCH");
        return v && v[0] == '1' && v[1] == '\0';
    }();
    return on;
}

struct FusedPlan {
    int SB, TB, n_bg, n_tb, tiles_per_tb, num_tiles, ring, n_items;
    size_t slot_bytes, ctl_bytes, total;
};

// A tile's 128 rows are SB streams x TB tokens of one layer.  Tiles go in the
// order (token block, layer, stream group), so a layer's weights are fetched
// once per token block; the ring holds three token blocks of records.
//
// Cost of a tile by its tokens, against one of 128 tokens: a shorter block means
// a smaller ring, whose records are read (and their lines overwritten) while
// they are still in L2, and shorter scan items; but the weights are fetched
// more often.  Measured, us: N = 32, 64 x 1000 tokens, TB = 128 1532, 64 1475,
// 32 1430, 16 1361; N = 64, 40 x 600 568, 561, 561 (of fewer tiles), 625;
// N = 128, 64 x 1024 3970, 3916, 4088; R = 0, 48 x 777 1645 (336 tiles a
// layer), 1608 (312), 1684 (300).
inline double tile_cost(int N, int R, int tb) {
    const int i = tb == 128 ? 0 : tb == 64 ? 1 : tb == 32 ? 2 : 3;
    static const double cost[4][4] = {{1.0, 0.96, 0.93, 0.90},     // N <= 32
                                      {1.0, 0.99, 1.04, 1.15},     // N = 64
                                      {1.0, 0.985, 1.01, 1.07},    // N = 128
                                      {1.0, 1.05, 1.15, 1.25}};    // N = 128, R = 0
    return cost[N <= 32 ? 0 : N <= 64 ? 1 : R > 0 ? 2 : 3][i];
}

// DRAM time of a layer, in tiles, when the weights do not stay in L2 from one
// token block to the next: the hidden states once and the weights once a block,
// against a tile's time at 0.78 of the bf16 peak or, for few columns, that of
// its hidden rows.
inline double layer_bytes_cost(int columns, int n_bg, int n_tb) {
    const double flop_bound = columns / 216.0;           // a tile's MMAs : its hidden rows
    return n_tb * (n_bg + columns / 128.0) / (flop_bound > 1.0 ? flop_bound : 1.0);
}
constexpr double kL2Bytes = 129e6;

// Tokens of a block: all of a shorter call; otherwise the cheapest by tiles a
// layer times a tile's cost, an N = 128 plan whose tiles do not pair up (see
// launch_fused_pair) counting 12 % more, and no less than the DRAM time of
// weights that L2 does not hold (94 layers, d = 4096, 296 MB of them, 13 streams
// x 200 tokens: blocks of 16 986 us, 32 811, 64 846, 128 859).  With fewer chains than about the scan
// warps (1,024), or rows short enough that a tile's GEMM takes less than its
// scan (d < 1024), the chains' steps bound the call, not its tiles, and longer
// items are better (N = 16, d = 256, 256 x 500: 327 us, with TB = 16 358).
// T = 0 gives the largest layout.
inline int block_tokens(const crc_problem& p, int T) {
    int tb = 128;
    if (T > 0 && T <= 64)
        while (tb > 1 && tb / 2 >= T) tb >>= 1;
    if (T <= 64 || p.d < 1024 || (long long)p.B * p.L < 1024) return tb;
    double best = 0.0;
    for (int c = 128; c >= 16; c >>= 1) {
        const int n_bg = (p.B + 128 / c - 1) / (128 / c);
        double cost = (double)n_bg * ((T + c - 1) / c) * tile_cost(p.N, p.R, c);
        if (p.N == 128 && n_bg % 2 != 0) cost *= 1.12;
        const int columns = (p.R > 0 ? 3 : 2) * p.N;
        if (2.0 * p.L * columns * p.d > kL2Bytes)
            cost = std::max(cost, layer_bytes_cost(columns, n_bg, (T + c - 1) / c));
        if (c == 128 || cost < best) {
            best = cost;
            tb = c;
        }
    }
    return tb;
}

inline FusedPlan fused_plan(const crc_problem& p, int T) {
    FusedPlan f;
    const int tb = block_tokens(p, T);
    f.TB = tb;
    f.SB = 128 / tb;
    f.n_bg = (p.B + f.SB - 1) / f.SB;
    f.tiles_per_tb = p.L * f.n_bg;
    f.n_tb = (T + f.TB - 1) / f.TB;
    f.num_tiles = f.n_tb * f.tiles_per_tb;
    f.ring = 3 * f.tiles_per_tb;
    if (T > 0) f.ring = std::min(f.ring, f.num_tiles);
    f.n_items = f.n_tb * p.L * p.B;
    const int NW = (p.N + 31) / 32;
    f.slot_bytes = (size_t)128 * 4 * (NW + p.N * (p.R > 0 ? 2 : 1));
    const size_t ctl = 256 + (size_t)4 * 3 * f.tiles_per_tb * 2 + (size_t)4 * p.B * p.L;
    f.ctl_bytes = (ctl + 255) & ~(size_t)255;
    f.total = f.ctl_bytes + (size_t)3 * f.tiles_per_tb * f.slot_bytes;
    return f;
}

// PAIR launches clusters of two CTAs (the GEMM on CTA pairs), cooperatively so
// that every CTA is resident; a device that refuses that launch gets the
// single-CTA kernel from then on (CRC_EUNSUPPORTED).
template <int NH, int H, int V, bool ALL_VALID, int KP, bool PAIR, bool TRACED>
int launch_fused_t(const crc_problem& p, const uint16_t* hidden, const uint16_t* w_cat, int T,
                   void* state, void* workspace, const crc_trace* trace,
                      cudaStream_t stream) {
    using Cfg = FusedCfg<NH, H, PAIR>;
    using RC = typename Cfg::RC;
    const FusedPlan f = fused_plan(p, T);
    if (PAIR && f.n_bg % 2 != 0) return CRC_EUNSUPPORTED;
    auto kern = fused_route_cache_kernel<NH, H, V, ALL_VALID, KP, PAIR, TRACED>;
    static PerDevice grids;                    // CTAs of the launch; -1: the device refuses it
    const int dev = current_device();
    const int grid = grids.get(dev, [&] {
        if (cuda_status(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             Cfg::SMEM_BYTES)))
            return 0;
        if (PAIR) {
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = 2;
            at[0].val.clusterDim.y = 1;
            at[0].val.clusterDim.z = 1;
            cudaLaunchConfig_t c = {};
            c.gridDim = dim3((unsigned)(sm_count() / 2 * 2));
            c.blockDim = dim3(Cfg::MAX_THREADS);
            c.dynamicSmemBytes = Cfg::SMEM_BYTES;
            c.attrs = at;
            c.numAttrs = 1;
            int ncl = 0;
            if (cuda_status(cudaOccupancyMaxActiveClusters(&ncl, (const void*)kern, &c))) return 0;
            return ncl > 0 ? std::min(2 * ncl, sm_count() / 2 * 2) : -1;
        }
        int per_sm = 0;
        if (cuda_status(cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                &per_sm, kern, Cfg::MAX_THREADS, Cfg::SMEM_BYTES)))
            return 0;
        return per_sm > 0 ? sm_count() : -1;
    });
    if (grid < 1) return CRC_EUNSUPPORTED;
    CUtensorMap mh, mw;
    if (!make_hidden_map(&mh, hidden, p.B, T, p.L, p.d, f.TB, f.SB)) return CRC_ECUDA;
    if (!make_weight_map(&mw, w_cat, p.L, 3 * NH, p.d, Cfg::B_BOX_ROWS)) return CRC_ECUDA;
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    if (const int rc = cuda_status(cudaMemsetAsync(ws, 0, f.ctl_bytes, stream))) return rc;
    FusedArgs a;
    a.state = static_cast<uint8_t*>(state);
    a.B = p.B;
    a.L = p.L;
    a.N = p.N;
    a.K = p.K;
    a.C = p.C;
    a.R = p.R;
    a.T = T;
    a.SB = f.SB;
    a.TB = f.TB;
    a.n_bg = f.n_bg;
    a.n_tb = f.n_tb;
    a.tiles_per_tb = f.tiles_per_tb;
    a.num_tiles = f.num_tiles;
    a.ring = f.ring;
    a.kblocks = (p.d + RC::BK - 1) / RC::BK;
    a.n_items = f.n_items;
    a.ctl = reinterpret_cast<uint32_t*>(ws);
    a.tile_done = reinterpret_cast<uint32_t*>(ws + 256);
    a.readers = a.tile_done + f.ring;
    a.prog = a.readers + f.ring;
    a.ring_base = ws + f.ctl_bytes;
    a.slot_bytes = f.slot_bytes;
    a.tr_miss = trace ? trace->misses_dev : nullptr;
    a.tr_pro = trace ? trace->proactive_dev : nullptr;
    a.tr_mid = trace ? trace->cache_mid_dev : nullptr;
    a.tr_after = trace ? trace->cache_after_dev : nullptr;
    a.tr_sel = trace ? trace->topk_set_dev : nullptr;
    void* args[] = {(void*)&mh, (void*)&mw, (void*)&a};
    const int threads = Cfg::threads_for(p.R, f.TB);
    cudaError_t e;
    if (PAIR) {
        cudaLaunchAttribute at[2];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 2;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        at[1].id = cudaLaunchAttributeCooperative;
        at[1].val.cooperative = 1;
        cudaLaunchConfig_t c = {};
        c.gridDim = dim3((unsigned)grid);
        c.blockDim = dim3(threads);
        c.dynamicSmemBytes = Cfg::SMEM_BYTES;
        c.stream = stream;
        c.attrs = at;
        // CRC_PLAIN_CLUSTER_LAUNCH=1 drops the cooperative attribute so that a
        // kernel profiler, which cannot replay a cooperative cluster launch,
        // can run the same kernel; the grid still fits the GPU at once (the
        // occupancy query above), and were it ever not co-resident, the bounded
        // waits would end the call with CRC_ETIMEOUT
        c.numAttrs = plain_cluster_launch() ? 1 : 2;
        {
            ProfScope prof(CRC_KERNEL_FUSED, stream);
            e = cudaLaunchKernelExC(&c, (const void*)kern, args);
        }
        if (cuda_status(e)) {
            grids.set(dev, -1);
            return CRC_EUNSUPPORTED;
        }
    } else {
        ProfScope prof(CRC_KERNEL_FUSED, stream);
        e = cudaLaunchCooperativeKernel((const void*)kern, grid, threads, args,
                                        Cfg::SMEM_BYTES, stream);
    }
    note_launch();
    return cuda_status(e);
}

// The GEMM on CTA pairs (N = 128: three heads, or two in update-only mode)
// when the tiles pair up; CRC_EUNSUPPORTED sends the call to one CTA per tile.
template <int NH, int H, int V, bool ALL_VALID, bool TRACED>
int launch_fused_pair(const crc_problem& p, const uint16_t* hidden, const uint16_t* w_cat, int T,
                      void* state, void* workspace, const crc_trace* trace,
                      cudaStream_t stream) {
    if constexpr (NH != 128) {
        return CRC_EUNSUPPORTED;
    } else {
        if (p.K <= 2)
            return launch_fused_t<NH, H, V, ALL_VALID, 2, true, TRACED>(p, hidden, w_cat, T,
                                                                        state, workspace, trace,
                                                                        stream);
        if (p.K <= 4)
            return launch_fused_t<NH, H, V, ALL_VALID, 4, true, TRACED>(p, hidden, w_cat, T,
                                                                        state, workspace, trace,
                                                                        stream);
        if (p.K <= 8)
            return launch_fused_t<NH, H, V, ALL_VALID, 8, true, TRACED>(p, hidden, w_cat, T,
                                                                        state, workspace, trace,
                                                                        stream);
        return CRC_EUNSUPPORTED;
    }
}

// Dispatch on heads (R > 0 needs the Spatio head) and the Top-K network width.
template <int NH, int V, bool ALL_VALID, bool TRACED>
int launch_fused_mode(const crc_problem& p, const uint16_t* hidden, const uint16_t* w_cat,
                       int T, void* state, void* workspace, const crc_trace* trace,
                       cudaStream_t stream) {
#define CRC_FUSED_KP(HV)                                                                      \
    {                                                                                         \
        const int rc = launch_fused_pair<NH, HV, V, ALL_VALID, TRACED>(p, hidden, w_cat, T,   \
                                                                       state, workspace,      \
                                                                       trace, stream);        \
        if (rc != CRC_EUNSUPPORTED) return rc;                                                \
    }                                                                                         \
    if (p.K <= 2)                                                                             \
        return launch_fused_t<NH, HV, V, ALL_VALID, 2, false, TRACED>(                        \
            p, hidden, w_cat, T, state, workspace, trace, stream);                            \
    if (p.K <= 4)                                                                             \
        return launch_fused_t<NH, HV, V, ALL_VALID, 4, false, TRACED>(                        \
            p, hidden, w_cat, T, state, workspace, trace, stream);                            \
    if (p.K <= 8)                                                                             \
        return launch_fused_t<NH, HV, V, ALL_VALID, 8, false, TRACED>(                        \
            p, hidden, w_cat, T, state, workspace, trace, stream);                            \
    return CRC_EUNSUPPORTED;
    if (p.R > 0) {
        CRC_FUSED_KP(3)
    } else {
        CRC_FUSED_KP(2)
    }
#undef CRC_FUSED_KP
}

// The kernel without trace writes unless the call asks for a trace array.
template <int NH, int V, bool ALL_VALID>
int launch_fused_for_n(const crc_problem& p, const uint16_t* hidden, const uint16_t* w_cat,
                       int T, void* state, void* workspace, const crc_trace* trace,
                       cudaStream_t stream) {
    return trace_wanted(trace)
               ? launch_fused_mode<NH, V, ALL_VALID, true>(p, hidden, w_cat, T, state, workspace,
                                                           trace, stream)
               : launch_fused_mode<NH, V, ALL_VALID, false>(p, hidden, w_cat, T, state, workspace,
                                                            nullptr, stream);
}

}  // namespace crc
