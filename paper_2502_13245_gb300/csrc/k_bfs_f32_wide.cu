// k_bfs_f32_wide.cu -- cluster expansion (k_bfs.cuh): fp32 indexes with rows of up to 2,048 bytes.
#include "k_bfs.cuh"

namespace rr {

rr_status launch_bfs_f32_wide(const BfsArgs &g, const BfsShape &s, cudaStream_t st) { return bfs_t<DT_F32, 4>(g, s, st); }

}  // namespace rr
