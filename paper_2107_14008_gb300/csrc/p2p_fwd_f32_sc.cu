// FP32 forward kernel, scalar streams, whole rows (its own translation unit
// so that the variants compile in parallel).
#include "fwd_f32_common.cuh"

namespace psr {
template int launch_fwd_f32_variant<false, kRowsWhole>(const FwdArgs&, int, size_t, cudaStream_t);
template const void* fwd_f32_kernel_ptr<false>(int, int, int, int);
}  // namespace psr
