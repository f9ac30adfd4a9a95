// FP32 forward kernel, scalar streams, heavy items on whole blocks (its own translation unit so that
// the variants compile in parallel).
#include "fwd_f32_common.cuh"

namespace psr {
template int launch_fwd_f32_variant<false, true>(const FwdArgs&, int, size_t, cudaStream_t);
}  // namespace psr
