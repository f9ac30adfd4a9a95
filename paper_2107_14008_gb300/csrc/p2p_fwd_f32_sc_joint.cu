// FP32 forward kernel, scalar streams, rows with parts on groups of warps (its own translation unit
// so that the variants compile in parallel).
#include "fwd_f32_common.cuh"

namespace psr {
template int launch_fwd_f32_variant<false, kRowsJoint>(const FwdArgs&, int, size_t, cudaStream_t);
}  // namespace psr
