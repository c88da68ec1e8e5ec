// knn_far_64.cu -- furthest-neighbour and range passes of the block search for dimension bucket DP = 64.
#include "probe.cuh"

namespace dt {
template int launch_far_seed<64>(const TileArgs&, int, int, cudaStream_t);
template int launch_far_cap<64>(const TileArgs&, int, int, float*, cudaStream_t);
template int launch_far_tile<64>(const TileArgs&, int, int, bool, int*, int, cudaStream_t);
template int launch_range_tile<64>(const TileArgs&, int, int*, int, cudaStream_t);
template int launch_probe_far<64>(const ProbeArgs&, cudaStream_t);
template int launch_probe_range<64>(const ProbeArgs&, cudaStream_t);
}  // namespace dt
