// knn_far_32.cu -- furthest-neighbour and range passes of the block search for dimension bucket DP = 32.
#include "probe.cuh"

namespace dt {
template int launch_far_seed<32>(const TileArgs&, int, int, cudaStream_t);
template int launch_far_cap<32>(const TileArgs&, int, int, float*, cudaStream_t);
template int launch_far_tile<32>(const TileArgs&, int, int, bool, int*, int, cudaStream_t);
template int launch_range_tile<32>(const TileArgs&, int, int*, int, cudaStream_t);
template int launch_probe_far<32>(const ProbeArgs&, cudaStream_t);
template int launch_probe_range<32>(const ProbeArgs&, cudaStream_t);
}  // namespace dt
