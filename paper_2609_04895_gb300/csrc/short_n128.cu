// Short-call route-and-cache instantiations for N = 128 experts per layer.
#include "short_launch.cuh"

namespace crc {

int launch_short_n128(const crc_problem& p, const uint16_t* hidden, const uint16_t* w_cat, int T,
                      void* state, const crc_trace* trace, bool persistent,
                      cudaStream_t stream) {
    return launch_short_for_n<128, 4, true>(p, hidden, w_cat, T, state, trace, persistent, stream);
}

}  // namespace crc
