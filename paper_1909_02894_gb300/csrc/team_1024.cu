// Radix-16 team passes over 1024-point lines.
#include "team_launch.cuh"

namespace dgb {
template cudaError_t launch_team<1024>(const LinePassArgs<float>&, cudaStream_t);
template cudaError_t launch_team_unsplit<1024>(const UnsplitArgs&, int, cudaStream_t);
int dgb_debug_flag_team_1024() { return dgb_take_debug_flag(); }
}  // namespace dgb
