// knn_tc_32.cu -- tensor-core BaseCase tiles for dimension bucket DP = 32.
#include "knn_tc.cuh"

namespace dt {
template int launch_tile_tc<32>(const TileArgs&, int, int, int, bool, int*, int, cudaStream_t);
template size_t tc_ops_row_bytes<32>(int);
template int launch_tc_ops<32>(const dtree_t*, int, int, void*, cudaStream_t);
}  // namespace dt
