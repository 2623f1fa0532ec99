// k_bfs_i8.cu -- cluster expansion (k_bfs.cuh): int8 indexes.
#include "k_bfs.cuh"

namespace rr {

rr_status launch_bfs_i8(const BfsArgs &g, const BfsShape &s, cudaStream_t st) { return bfs_t<DT_I8, 1>(g, s, st); }

}  // namespace rr
