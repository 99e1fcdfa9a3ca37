// Radix-16 team passes over 2048-point lines.
#include "team_launch.cuh"

namespace dgb {
template cudaError_t launch_team<2048>(const LinePassArgs<float>&, cudaStream_t);
template cudaError_t launch_team_unsplit<2048>(const UnsplitArgs&, int, cudaStream_t);
int dgb_debug_flag_team_2048() { return dgb_take_debug_flag(); }
}  // namespace dgb
