// Fused line pass, complex64 state (FP32 arithmetic, FP64-derived tables).
#include "launch_impl.cuh"

namespace dgb {
template cudaError_t launch_line_pass<float>(const LinePassArgs<float>&, int, int, cudaStream_t);
template int line_pass_radix<float>(int);
template int line_pass_radix_alt<float>(int);
template int line_pass_radix_small<float>(int, int);

int dgb_debug_flag_c64() { return dgb_take_debug_flag(); }
}  // namespace dgb
