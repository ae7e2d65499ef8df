// Small problems in one cooperative launch (small.cuh), half messages.
#include "small.cuh"

namespace mld {

bool small_decode_f16(mld_decoder *d, int W, int32_t batch, int32_t iters, bool et, bool hard1, int32_t *iters_out,
                      uint8_t *conv_out, int sm_count, cudaStream_t st, bool soft) {
    switch (W) {
        case 8: return launch_small<__half, 8>(d, batch, iters, et, hard1, iters_out, conv_out, sm_count, st, soft);
        case 16: return launch_small<__half, 16>(d, batch, iters, et, hard1, iters_out, conv_out, sm_count, st, soft);
        case 32: return launch_small<__half, 32>(d, batch, iters, et, hard1, iters_out, conv_out, sm_count, st, soft);
        default: return launch_small<__half, 64>(d, batch, iters, et, hard1, iters_out, conv_out, sm_count, st, soft);
    }
}

}  // namespace mld
