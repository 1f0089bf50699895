// The streaming form's first launch for 8-bit codes (stream_kernel.cuh; one
// text, or a batch), compiled apart so that the forms build in parallel.
#include "stream_kernel.cuh"

namespace pfac {
namespace strm {

cudaError_t launch_stream8(OutMode mode, const StreamParams &p, uint32_t grid, uint32_t smem, int max_smem,
                           cudaStream_t stream) {
    switch (mode) {
        case OUT_DENSE: return launch_form<pfac_stream8<OUT_DENSE>, 8>(p, grid, smem, max_smem, stream);
        case OUT_COUNT: return launch_form<pfac_stream8<OUT_COUNT>, 8>(p, grid, smem, max_smem, stream);
        case OUT_BITS: return launch_form<pfac_stream8<OUT_BITS>, 8>(p, grid, smem, max_smem, stream);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_stream8_multi(OutMode mode, const StreamMulti &mp, uint32_t grid, uint32_t smem, int max_smem,
                                 cudaStream_t stream) {
    switch (mode) {
        case OUT_DENSE: return launch_form<pfac_stream8_multi<OUT_DENSE>, 8>(mp, grid, smem, max_smem, stream);
        case OUT_BITS: return launch_form<pfac_stream8_multi<OUT_BITS>, 8>(mp, grid, smem, max_smem, stream);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace strm
}  // namespace pfac
