// k_bfs_f32.cu -- cluster expansion (k_bfs.cuh): fp32 indexes with rows of up to 1,024 bytes.
#include "k_bfs.cuh"

namespace rr {

rr_status launch_bfs_f32(const BfsArgs &g, const BfsShape &s, cudaStream_t st) {
    if (g.s.row_chunks <= 32) return bfs_t<DT_F32, 1>(g, s, st);
    return bfs_t<DT_F32, 2>(g, s, st);
}

}  // namespace rr
