// The streaming form's first launch for 8-bit codes (stream_kernel.cuh; one
// text, or a batch), compiled apart so that the forms build in parallel.
#include "stream_kernel.cuh"

namespace pfac {
namespace strm {

cudaError_t launch_stream8(OutMode mode, const StreamParams &p, uint32_t grid, uint32_t smem, int max_smem,
                           cudaStream_t stream) {
    switch (mode) {
        case OUT_DENSE: return launch_form<pfac_stream8<OUT_DENSE>>(p, grid, kBlock8, smem, max_smem, stream);
        case OUT_COUNT: return launch_form<pfac_stream8<OUT_COUNT>>(p, grid, kBlock8, smem, max_smem, stream);
        case OUT_BITS: return launch_form<pfac_stream8<OUT_BITS>>(p, grid, kBlock8, smem, max_smem, stream);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_stream8_multi(OutMode mode, const StreamMulti &mp, uint32_t grid, uint32_t smem, int max_smem,
                                 cudaStream_t stream, bool next) {
    switch (mode) {
        case OUT_DENSE: return launch_form<pfac_stream8_multi<OUT_DENSE>>(mp, grid, kBlock8Multi, smem, max_smem, stream, next);
        case OUT_BITS: return launch_form<pfac_stream8_multi<OUT_BITS>>(mp, grid, kBlock8Multi, smem, max_smem, stream, next);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace strm
}  // namespace pfac
