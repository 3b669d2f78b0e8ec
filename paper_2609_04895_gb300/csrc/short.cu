// Short-call route-and-cache: which calls it takes, and the dispatch on N.
#include "short_launch.cuh"

namespace crc {

int launch_short_n128(const crc_problem& p, const uint16_t* hidden, const uint16_t* w_cat, int T,
                      void* state, const crc_trace* trace, cudaStream_t stream);

// Where a call is faster on the short-call kernel than on the persistent fused
// one (times in us, persistent / short, traced calls on one GB300):
//  - one or two tokens, any batch: the persistent kernel's tiles are then one
//    layer's whole work and its scan items one step long.  N = 128, d = 2048,
//    48 layers: T = 1, B = 64 56 / 31, B = 1024 348 / 152; N = 32: B = 1024
//    150 / 73; d = 4096: T = 2, B = 256 243 / 222.
//  - up to four unless d is large, when the hidden rows that the heads' CTAs
//    read again cost more (T = 4, B = 128: d = 2048 109 / 95, d = 4096
//    197 / 229).
//  - up to 64 tokens when every CTA is resident at once, two an SM (three for
//    N = 128): with a second wave the chains' steps, which take most of such a
//    call, come twice (N = 128: T = 24, B = 13 91 / 63; T = 16, B = 16 60 / 47;
//    T = 16, B = 64 128 / 154).  Untraced calls of up to 32 experts only to 32
//    tokens (T = 64, B = 1: 57 / 57), longer ones not at all: the persistent
//    kernel runs several tiles' chains side by side.
static bool takes(const crc_problem& p, int T, bool traced) {
    if (T <= 2) return true;
    if (T <= 4 && p.d <= 3072) return true;
    if (T > (traced || p.N > 32 ? 64 : 32)) return false;
    const int SB = std::min(p.B, 128 / T);
    const long long ctas = (long long)p.L * ((p.B + SB - 1) / SB) * (p.R > 0 ? 3 : 2);
    return ctas <= (long long)sm_count() * (p.N == 128 ? 3 : 2);
}

int launch_short(const crc_problem& p, const uint16_t* hidden, const uint16_t* w_cat, int T,
                 void* state, const crc_trace* trace, cudaStream_t stream) {
    if (p.K > 8 || !takes(p, T, trace_wanted(trace))) return CRC_EUNSUPPORTED;
    switch (p.N) {
        case 16: return launch_short_for_n<16, 1, false>(p, hidden, w_cat, T, state, trace, stream);
        case 32: return launch_short_for_n<32, 1, true>(p, hidden, w_cat, T, state, trace, stream);
        case 64: return launch_short_for_n<64, 2, true>(p, hidden, w_cat, T, state, trace, stream);
        case 128: return launch_short_n128(p, hidden, w_cat, T, state, trace, stream);
        default: return CRC_EUNSUPPORTED;
    }
}

}  // namespace crc
