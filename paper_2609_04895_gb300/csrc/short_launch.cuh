// Host side of the short-call kernel: its plan, tensor maps and launch.
#pragma once

#include <algorithm>

#include "crc_internal.h"
#include "short_call.cuh"

namespace crc {

// Shared memory a CTA may take so that two (twelve warps each) or three (eight
// warps each) fit an SM: 80 registers a thread allow both.  Three when the
// call has more CTAs than two an SM: they wait on their chains' steps, and
// more of them overlap.
constexpr int kShortSmem2 = 113 * 1024;
constexpr int kShortSmem3 = 75 * 1024;

// Any array of the trace that the fused kernels write.
inline bool trace_wanted(const crc_trace* t) {
    return t && (t->misses_dev || t->proactive_dev || t->cache_mid_dev || t->cache_after_dev ||
                 t->topk_set_dev);
}

template <int NH, int V, bool ALL_VALID, bool TRACED>
int launch_short_t(const crc_problem& p, const uint16_t* hidden, const uint16_t* w_cat, int T,
                   void* state, const crc_trace* trace, cudaStream_t stream) {
    using Cfg = ShortCfg<NH>;
    ShortArgs a;
    a.state = static_cast<uint8_t*>(state);
    a.B = p.B;
    a.L = p.L;
    a.N = p.N;
    a.K = p.K;
    a.C = p.C;
    a.R = p.R;
    a.T = T;
    a.SB = std::min(p.B, 128 / T);
    a.n_bg = (p.B + a.SB - 1) / a.SB;
    a.kblocks = (p.d + Cfg::BK - 1) / Cfg::BK;
    const int H = p.R > 0 ? 3 : 2;
    const int grid = p.L * a.n_bg * H;
    const int rows = a.SB * T;
    a.a_bytes = rows * 128;
    a.stage_bytes = ((a.a_bytes + 1023) & ~1023) + Cfg::W_BYTES;
    // the MMA reads 128 rows from the start of a stage, whatever follows the box
    const int overrun = std::max(0, 128 * 128 - a.stage_bytes);
    // the probabilities take the stages' place, behind them the Top-K bytes of a third
    // (half) of the streams, and their traced sets, misses and loads
    const int own_rows = (a.SB + H - 1) / H * T;
    a.sel_at = (rows * Cfg::ROW_FLOATS * 4 + 15) & ~15;
    a.tr_at = a.sel_at + own_rows * 32;
    const int after = a.tr_at + (TRACED ? own_rows * 34 : 0);
    const int fixed = 1024 + Cfg::TAIL_BYTES;
    const bool three = grid > 2 * sm_count() && fixed + after <= kShortSmem3;
    const int room = (three ? kShortSmem3 : kShortSmem2) - fixed - overrun;
    a.stages = std::max(1, std::min({kShortMaxStages, a.kblocks, room / a.stage_bytes}));
    a.tail = (std::max(a.stages * a.stage_bytes + overrun, after) + 1023) & ~1023;
    const int smem = fixed + a.tail;
    const int threads = three ? 256 : Cfg::MAX_THREADS;
    a.tr_miss = trace ? trace->misses_dev : nullptr;
    a.tr_pro = trace ? trace->proactive_dev : nullptr;
    a.tr_mid = trace ? trace->cache_mid_dev : nullptr;
    a.tr_after = trace ? trace->cache_after_dev : nullptr;
    a.tr_sel = trace ? trace->topk_set_dev : nullptr;
    auto kern = short_call_kernel<NH, V, ALL_VALID, TRACED>;
    static PerDevice ready;
    const int up = ready.get(current_device(), [&] {
        return cuda_status(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                kShortSmem2)) == CRC_OK;
    });
    if (!up) return CRC_ECUDA;
    CUtensorMap mh, mw;
    if (!make_hidden_map(&mh, hidden, p.B, T, p.L, p.d, T, a.SB)) return CRC_ECUDA;
    if (!make_weight_map(&mw, w_cat, p.L, 3 * NH, p.d, NH)) return CRC_ECUDA;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)H;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3((unsigned)grid);
    c.blockDim = dim3((unsigned)threads);
    c.dynamicSmemBytes = (size_t)smem;
    c.stream = stream;
    c.attrs = at;
    c.numAttrs = 1;
    void* args[] = {(void*)&mh, (void*)&mw, (void*)&a};
    cudaError_t e;
    {
        ProfScope prof(CRC_KERNEL_SHORT, stream);
        e = cudaLaunchKernelExC(&c, (const void*)kern, args);
    }
    note_launch();
    return cuda_status(e);
}

template <int NH, int V, bool ALL_VALID>
int launch_short_for_n(const crc_problem& p, const uint16_t* hidden, const uint16_t* w_cat, int T,
                       void* state, const crc_trace* trace, cudaStream_t stream) {
    return trace_wanted(trace)
               ? launch_short_t<NH, V, ALL_VALID, true>(p, hidden, w_cat, T, state, trace, stream)
               : launch_short_t<NH, V, ALL_VALID, false>(p, hidden, w_cat, T, state, nullptr,
                                                         stream);
}

}  // namespace crc
