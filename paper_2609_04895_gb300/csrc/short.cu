// Short-call route-and-cache: the dispatch on N (the launcher knows which calls it takes).
#include "short_launch.cuh"

namespace crc {

int launch_short_n128(const crc_problem& p, const uint16_t* hidden, const uint16_t* w_cat, int T,
                      void* state, const crc_trace* trace, bool persistent,
                      cudaStream_t stream);

int launch_short(const crc_problem& p, const uint16_t* hidden, const uint16_t* w_cat, int T,
                 void* state, const crc_trace* trace, bool persistent, cudaStream_t stream) {
    if (p.K > 8 || T > 64) return CRC_EUNSUPPORTED;
    switch (p.N) {
        case 16:
            return launch_short_for_n<16, 1, false>(p, hidden, w_cat, T, state, trace, persistent,
                                                    stream);
        case 32:
            return launch_short_for_n<32, 1, true>(p, hidden, w_cat, T, state, trace, persistent,
                                                   stream);
        case 64:
            return launch_short_for_n<64, 2, true>(p, hidden, w_cat, T, state, trace, persistent,
                                                   stream);
        case 128: return launch_short_n128(p, hidden, w_cat, T, state, trace, persistent, stream);
        default: return CRC_EUNSUPPORTED;
    }
}

}  // namespace crc
