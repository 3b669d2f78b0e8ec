// Host launcher of the router-heads kernel: tensor maps, tile plan, dispatch.
#include <cudaTypedefs.h>

#include <mutex>

#include "crc_internal.h"
#include "router_gemm.cuh"
#include "router_pair.cuh"

namespace crc {

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000,
                                             cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    return fn;
}

// hidden [B][T_total][L][d] bf16 viewed as a 4-D tensor (d, L, T, B); a box is
// 64 hidden elements (one 128-byte swizzle row) x 1 layer x TB tokens x SB streams.
bool make_hidden_map(CUtensorMap* m, const uint16_t* hidden, int B, int T_total, int L, int d,
                     int TB, int SB) {
    auto enc = encode_fn();
    if (!enc) return false;
    cuuint64_t dims[4] = {(cuuint64_t)d, (cuuint64_t)L, (cuuint64_t)T_total, (cuuint64_t)B};
    cuuint64_t strides[3] = {(cuuint64_t)d * 2, (cuuint64_t)L * d * 2,
                             (cuuint64_t)T_total * L * d * 2};
    cuuint32_t box[4] = {64, 1, (cuuint32_t)TB, (cuuint32_t)SB};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<uint16_t*>(hidden), dims,
               strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// W_cat [L][3N][d] bf16 viewed as (d, 3N, L); a box is 64 x rows x 1 layer.
bool make_weight_map(CUtensorMap* m, const uint16_t* w, int L, int N3, int d, int rows) {
    auto enc = encode_fn();
    if (!enc) return false;
    cuuint64_t dims[3] = {(cuuint64_t)d, (cuuint64_t)N3, (cuuint64_t)L};
    cuuint64_t strides[2] = {(cuuint64_t)d * 2, (cuuint64_t)N3 * d * 2};
    cuuint32_t box[3] = {64, (cuuint32_t)rows, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<uint16_t*>(w), dims, strides,
               box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// scores [B][T_ext][L][3][NH] fp32 viewed as (NH, 3, L, T, B); a store box is
// 32 scores x 1 head x 1 layer x TBq tokens x SBq streams (32 rows, 128-byte rows).
bool make_scores_map(CUtensorMap* m, float* scores, int B, int T_ext, int L, int NH, int TBq,
                     int SBq) {
    auto enc = encode_fn();
    if (!enc) return false;
    cuuint64_t dims[5] = {(cuuint64_t)NH, 3, (cuuint64_t)L, (cuuint64_t)T_ext, (cuuint64_t)B};
    cuuint64_t strides[4] = {(cuuint64_t)NH * 4, (cuuint64_t)3 * NH * 4,
                             (cuuint64_t)L * 3 * NH * 4, (cuuint64_t)T_ext * L * 3 * NH * 4};
    cuuint32_t box[5] = {32, 1, 1, (cuuint32_t)TBq, (cuuint32_t)SBq};
    cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 5, scores, dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

namespace {

// The launch on CTA pairs.  A layer's tiles are paired in order; an odd last
// one has an idle partner.  What decides is the rounds of tiles that an SM runs:
// a pair's round takes 0.86 to 0.96 of a single CTA's for d >= 2048 (0.87 to 0.92
// at d = 7168), so pairs pay unless idle partners add more than one round in
// sixteen.  Us, single / pairs, three heads: 48 layers of 9 tiles, 3 rounds
// against 4, 82 / 95; of 15, 5 against 6, 129 / 139; 94 layers of 27, 17 against
// 18, 425 / 419.  Shorter rows are bound by the epilogue and gain nothing
// (d = 1024, equal rounds: 0.95 to 1.06), and a call of one round has the
// cluster's set-up to make up for as well (d = 2048 0.94 to 1.08, d = 1024 1.00
// to 1.09, d = 4096 0.87 to 1.02).  CRC_EUNSUPPORTED: the single-CTA kernel
// takes the call.
template <int H>
int launch_router_pair(const crc_problem& p, const uint16_t* w_cat, const CUtensorMap& mh,
                       const CUtensorMap& ms, const RouterArgs& a, cudaStream_t stream) {
    using Cfg = RouterPairCfg<H>;
    RouterPairArgs pa;
    pa.r = a;
    const int tiles = a.n_sb * a.n_tb;
    pa.pairs_per_layer = (tiles + 1) / 2;
    pa.num_pairs = p.L * pa.pairs_per_layer;
    const int sms = sm_count(), pairs = sms / 2;
    const int rounds = (a.num_tiles + sms - 1) / sms;
    const int pair_rounds = pairs > 0 ? (pa.num_pairs + pairs - 1) / pairs : 0;
    if (p.d < (rounds > 1 ? 2048 : 4096) || pairs < 1 || 15ll * pair_rounds > 16ll * rounds)
        return CRC_EUNSUPPORTED;
    auto kern = router_pair_kernel<H>;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3((unsigned)(sm_count() / 2 * 2));
    c.blockDim = dim3(Cfg::THREADS);
    c.dynamicSmemBytes = Cfg::SMEM_BYTES;
    c.stream = stream;
    c.attrs = at;
    c.numAttrs = 1;
    static PerDevice resident;                 // clusters that fit the GPU at once
    const int fit = resident.get(current_device(), [&] {
        int n = 0;
        if (cuda_status(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             Cfg::SMEM_BYTES)) ||
            cuda_status(cudaOccupancyMaxActiveClusters(&n, (const void*)kern, &c)))
            return 0;
        return n > 0 ? n : -1;
    });
    if (fit < 1) return CRC_EUNSUPPORTED;
    c.gridDim = dim3((unsigned)(2 * (pa.num_pairs < fit ? pa.num_pairs : fit)));
    CUtensorMap mw;
    if (!make_weight_map(&mw, w_cat, p.L, 3 * Cfg::NH, p.d, Cfg::W_ROWS)) return CRC_ECUDA;
    void* args[] = {(void*)&mh, (void*)&mw, (void*)&ms, (void*)&pa};
    cudaError_t e;
    {
        ProfScope prof(CRC_KERNEL_ROUTER, stream);
        e = cudaLaunchKernelExC(&c, (const void*)kern, args);
    }
    note_launch();
    return cuda_status(e);
}

template <int NH, int H>
int launch_router_t(const crc_problem& p, const uint16_t* hidden, int T_total, int t_begin,
                    int T_ext, const uint16_t* w_cat, float* scores, uint32_t* err,
                    cudaStream_t stream) {
    using Cfg = RouterCfg<NH, H>;
    int TB = 1;
    while (TB < T_ext && TB < Cfg::BM) TB <<= 1;
    const int SB = Cfg::BM / TB;
    CUtensorMap mh, mw;
    if (!make_hidden_map(&mh, hidden, p.B, T_total, p.L, p.d, TB, SB)) return CRC_ECUDA;
    if (!make_weight_map(&mw, w_cat, p.L, 3 * NH, p.d, Cfg::B_BOX_ROWS)) return CRC_ECUDA;
    CUtensorMap ms = mh;   // unused when a head is narrower than one 32-score store box
    if (Cfg::TMA_STORE) {
        const int TBq = TB < 32 ? TB : 32;
        if (!make_scores_map(&ms, scores, p.B, T_ext, p.L, NH, TBq, 32 / TBq)) return CRC_ECUDA;
    }
    RouterArgs a;
    a.scores = scores;
    a.err = err;
    a.B = p.B;
    a.L = p.L;
    a.d = p.d;
    a.t_begin = t_begin;
    a.T_ext = T_ext;
    a.SB = SB;
    a.TB = TB;
    a.n_sb = (p.B + SB - 1) / SB;
    a.n_tb = (T_ext + TB - 1) / TB;
    a.num_tiles = p.L * a.n_sb * a.n_tb;
    a.kblocks = (p.d + Cfg::BK - 1) / Cfg::BK;
    static PerDevice ready;
    const int up = ready.get(current_device(), [&] {
        return cuda_status(cudaFuncSetAttribute(router_heads_kernel<NH, H>,
                                                cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                Cfg::SMEM_BYTES)) == CRC_OK;
    });
    if (!up) return CRC_ECUDA;
    if constexpr (NH == 128) {
        const int rc = launch_router_pair<H>(p, w_cat, mh, ms, a, stream);
        if (rc != CRC_EUNSUPPORTED) return rc;
    }
    const int grid = a.num_tiles < sm_count() ? a.num_tiles : sm_count();
    {
        ProfScope prof(CRC_KERNEL_ROUTER, stream);
        router_heads_kernel<NH, H><<<grid, Cfg::THREADS, Cfg::SMEM_BYTES, stream>>>(mh, mw, ms, a);
    }
    note_launch();
    return cuda_status(cudaGetLastError());
}

}  // namespace

int launch_router(const crc_problem& p, const uint16_t* hidden, int T_total, int t_begin,
                  int T_ext, const uint16_t* w_cat, int heads, float* scores,
                  uint32_t* err_word, cudaStream_t stream) {
    if (T_ext <= 0) return CRC_OK;
#define CRC_ROUTER_CASE(NHV)                                                                \
    case NHV:                                                                               \
        return heads == 3 ? launch_router_t<NHV, 3>(p, hidden, T_total, t_begin, T_ext,     \
                                                    w_cat, scores, err_word, stream)        \
                          : launch_router_t<NHV, 2>(p, hidden, T_total, t_begin, T_ext,     \
                                                    w_cat, scores, err_word, stream);
    switch (p.N) {
        CRC_ROUTER_CASE(16)
        CRC_ROUTER_CASE(32)
        CRC_ROUTER_CASE(64)
        CRC_ROUTER_CASE(128)
        default:
            return CRC_EUNSUPPORTED;
    }
#undef CRC_ROUTER_CASE
}

}  // namespace crc
