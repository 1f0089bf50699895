// The streaming form's first launch for 2-bit codes (stream_kernel.cuh; one
// text, or a batch), compiled apart so that the forms build in parallel.
#include "stream_kernel.cuh"

namespace pfac {
namespace strm {

template <int S>
static cudaError_t launch_step(OutMode mode, const StreamParams &p, uint32_t grid, uint32_t smem, int max_smem,
                               cudaStream_t stream) {
    switch (mode) {
        case OUT_DENSE: return launch_form<pfac_stream2<S, OUT_DENSE>>(p, grid, kBlock2, smem, max_smem, stream);
        case OUT_COUNT: return launch_form<pfac_stream2<S, OUT_COUNT>>(p, grid, kBlock2, smem, max_smem, stream);
        case OUT_BITS: return launch_form<pfac_stream2<S, OUT_BITS>>(p, grid, kBlock2, smem, max_smem, stream);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_stream2(OutMode mode, const StreamParams &p, uint32_t step, uint32_t grid, uint32_t smem,
                           int max_smem, cudaStream_t stream) {
    switch (step) {
        case 1: return launch_step<1>(mode, p, grid, smem, max_smem, stream);
        case 2: return launch_step<2>(mode, p, grid, smem, max_smem, stream);
        case 4: return launch_step<4>(mode, p, grid, smem, max_smem, stream);
        default: return cudaErrorInvalidValue;
    }
}

template <int S>
static cudaError_t launch_multi(OutMode mode, const StreamMulti &mp, uint32_t grid, uint32_t smem, int max_smem,
                                cudaStream_t stream, bool next) {
    switch (mode) {
        case OUT_DENSE: return launch_form<pfac_stream2_multi<S, OUT_DENSE>>(mp, grid, kBlock2, smem, max_smem, stream, next);
        case OUT_BITS: return launch_form<pfac_stream2_multi<S, OUT_BITS>>(mp, grid, kBlock2, smem, max_smem, stream, next);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_stream2_multi(OutMode mode, const StreamMulti &mp, uint32_t step, uint32_t grid, uint32_t smem,
                                 int max_smem, cudaStream_t stream, bool next) {
    switch (step) {
        case 1: return launch_multi<1>(mode, mp, grid, smem, max_smem, stream, next);
        case 2: return launch_multi<2>(mode, mp, grid, smem, max_smem, stream, next);
        case 4: return launch_multi<4>(mode, mp, grid, smem, max_smem, stream, next);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace strm
}  // namespace pfac
