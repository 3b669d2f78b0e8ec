// Host side of the short-call kernel: its plan, tensor maps and launch.
#pragma once

#include <algorithm>

#include "crc_internal.h"
#include "short_call.cuh"

namespace crc {

// Shared memory a CTA may take so that two (twelve warps each) or three (eight
// warps each) fit an SM: 80 registers a thread allow both.
constexpr int kShortSmem2 = 113 * 1024;
constexpr int kShortSmem3 = 75 * 1024;

// Where a call is faster on the short-call kernel than on the persistent fused
// one, by the waves of clusters it would run in with two CTAs an SM and with
// three (times in us, persistent / short, traced calls on one GB300):
//  - one or two tokens: the persistent kernel's tiles are then one layer's whole
//    work and its scan items one step long.  N = 128, d = 2048, 48 layers: T = 1,
//    B = 64 56 / 31, B = 1024 348 / 152; N = 32: B = 1024 150 / 73; d = 4096:
//    T = 2, B = 256 243 / 222.  Not two tokens of wide rows in several waves,
//    when the hidden rows that the heads' CTAs read again cost more (N = 128,
//    d = 7168, T = 2, untraced: B = 128 140 / 118 in one wave, B = 200 171 / 201,
//    B = 600 384 / 493).
//  - up to four unless d is large, for the same reason (T = 4, B = 128:
//    d = 2048 109 / 95, d = 4096 197 / 229), nor four tokens of 128 experts in
//    more than three waves (T = 4, B = 300, untraced: 152 / 162).
//  - up to 64 tokens when every cluster is resident at once, two CTAs an SM
//    (three for N = 128): with a second wave the chains' steps, which take most
//    of such a call, come twice (N = 128: T = 24, B = 13 91 / 63; T = 16, B = 16
//    60 / 47; T = 16, B = 64 128 / 154).  Untraced calls of up to 32 experts only
//    to 32 tokens (T = 64, B = 1: 57 / 57), longer ones not at all: the
//    persistent kernel runs several tiles' chains side by side.
// Without room for the persistent kernel the choice is the router's and the
// scan's launches, a chunk of tokens at a time: up to two tokens, and four of
// rows that are not wide, are then taken in any number of waves.
inline bool short_call_takes(const crc_problem& p, int T, bool traced, bool persistent,
                             int waves2, int waves3) {
    const bool one_wave = waves2 <= 1 || (p.N == 128 && waves3 <= 1);
    if (T <= 1) return true;
    if (!persistent && (T <= 2 || (T <= 4 && p.d <= 3072))) return true;
    if (T <= 2) return one_wave || p.N < 128 || p.d <= 4096;
    if (T <= 4 && p.d <= 3072) return T <= 3 || p.N < 128 || waves2 <= 3;
    return T <= (traced || p.N > 32 ? 64 : 32) && one_wave;
}

template <int NH, int V, bool ALL_VALID, bool TRACED>
int launch_short_t(const crc_problem& p, const uint16_t* hidden, const uint16_t* w_cat, int T,
                   void* state, const crc_trace* trace, bool persistent, cudaStream_t stream) {
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
    // Waves of clusters.  Clusters of three leave a twentieth of the SMs' places
    // empty: with three CTAs an SM 144 of them run in one wave, 150 in two.
    const int places = std::max(1, sm_count() * 19 / 20);
    const int waves2 = (grid + 2 * places - 1) / (2 * places);
    const int waves3 =
        fixed + after <= kShortSmem3 ? (grid + 3 * places - 1) / (3 * places) : waves2;
    if (!short_call_takes(p, T, TRACED, persistent, waves2, waves3)) return CRC_EUNSUPPORTED;
    // Three CTAs an SM when that saves enough waves: they share the SM's loads,
    // so a wave takes 1.3 to 1.45 times one of two (1.6 for N = 64, whose three
    // have fewer bytes in flight).  One token, us, two / three an SM: N = 128,
    // d = 2048, B = 300, waves 2 / 1 65 / 50; B = 400, 2 / 2 70 / 84; B = 600,
    // 3 / 2 100 / 93; N = 64, d = 5120, B = 400, 2 / 1 73 / 67; B = 600, 2 / 2
    // 83 / 122; B = 1024, 3 / 2 128 / 139.
    const bool three = NH == 64 ? 8 * waves3 <= 5 * waves2 : 4 * waves3 <= 3 * waves2;
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
                       void* state, const crc_trace* trace, bool persistent,
                       cudaStream_t stream) {
    return trace_wanted(trace)
               ? launch_short_t<NH, V, ALL_VALID, true>(p, hidden, w_cat, T, state, trace,
                                                        persistent, stream)
               : launch_short_t<NH, V, ALL_VALID, false>(p, hidden, w_cat, T, state, nullptr,
                                                         persistent, stream);
}

}  // namespace crc
