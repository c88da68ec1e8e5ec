// knn_far_8.cu -- furthest-neighbour passes of the block search for dimension bucket DP = 8.
#include "knn_tc.cuh"

namespace dt {
template int launch_far_seed<8>(const TileArgs&, int, int, cudaStream_t);
template int launch_far_cap<8>(const TileArgs&, int, int, float*, cudaStream_t);
template int launch_far_tile<8>(const TileArgs&, int, int, bool, int*, int, cudaStream_t);
}  // namespace dt
