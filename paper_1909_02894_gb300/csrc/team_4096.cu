// Radix-16 team passes over 4096-point lines.
#include "team_launch.cuh"

namespace dgb {
template cudaError_t launch_team<4096>(const LinePassArgs<float>&, cudaStream_t);
template cudaError_t launch_team_unsplit<4096>(const UnsplitArgs&, int, cudaStream_t);
int dgb_debug_flag_team_4096() { return dgb_take_debug_flag(); }
}  // namespace dgb
