// Fused line pass, complex128 state (FP64 arithmetic).
#include "launch_impl.cuh"

namespace dgb {
template cudaError_t launch_line_pass<double>(const LinePassArgs<double>&, int, int, cudaStream_t);
template int line_pass_radix<double>(int);
template int line_pass_radix_alt<double>(int);
template int line_pass_radix_small<double>(int, int);

int dgb_debug_flag_c128() { return dgb_take_debug_flag(); }
}  // namespace dgb
