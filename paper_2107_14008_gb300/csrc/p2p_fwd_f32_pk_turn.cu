// FP32 forward kernel, packed pairs of the core form, rows with parts on one warp (its own translation unit
// so that the variants compile in parallel).
#include "fwd_f32_common.cuh"

namespace psr {
template int launch_fwd_f32_variant<true, kRowsInTurn>(const FwdArgs&, int, size_t, cudaStream_t);
}  // namespace psr
