// k_bfs_u8.cu -- cluster expansion (k_bfs.cuh): uint8 indexes, the launch shape and the dispatch.
#include <algorithm>

#include "k_bfs.cuh"

namespace rr {

rr_status launch_bfs_u8(const BfsArgs &g, const BfsShape &s, cudaStream_t st) { return bfs_t<DT_U8, 1>(g, s, st); }
rr_status launch_bfs_i8(const BfsArgs &g, const BfsShape &s, cudaStream_t st);
rr_status launch_bfs_f32(const BfsArgs &g, const BfsShape &s, cudaStream_t st);
rr_status launch_bfs_f32_wide(const BfsArgs &g, const BfsShape &s, cudaStream_t st);

bool bfs_shape(int64_t n, int64_t nq, BfsShape *s) {
    constexpr size_t kSmem = 227 * 1024;
    const size_t words = (size_t)((n + 31) / 32);
    s->cl_log2 = 0;
    s->threads = kBfsThreads;
    const size_t most = (kSmem - kCtlBytes - kBfsThreads / 32 * kWarpBytes) / 16 * 4;
    while (((words + ((size_t)1 << s->cl_log2) - 1) >> s->cl_log2) > most) s->cl_log2++;
    // beyond four CTAs too few queries are resident: at 10^7 points (eight) 2,267 queries with 11.1 M results took
    // 7.1 ms against 5.6 in the two-pass levels, at 5 * 10^6 (four) 2,286 with 12.6 M 3.8 against 5.7
    if (s->cl_log2 > 2) return false;
    s->bm_words = (int)(((((words + ((size_t)1 << s->cl_log2) - 1) >> s->cl_log2)) + 3) / 4 * 4);
    // small bitmaps: two CTAs of half the threads an SM, so one query's barriers overlap another's work
    if (s->cl_log2 == 0 && (size_t)s->bm_words * 4 <= 96 * 1024 && nq > 152) s->threads = kBfsThreads / 2;
    s->smem = (size_t)s->bm_words * 4 + (size_t)(s->threads / 32) * kWarpBytes + kCtlBytes;
    s->clusters = (int)std::max<int64_t>(1, std::min<int64_t>(nq, (152 * (kBfsThreads / s->threads)) >> s->cl_log2));
    s->fcap = (uint32_t)std::min<int64_t>(n, (int64_t)1 << (17 + s->cl_log2));
    return true;
}

size_t bfs_front_bytes(const BfsShape &s) { return (size_t)2 * s.fcap * 4; }

int64_t bfs_list_slack(const BfsShape &s) {
    return ((int64_t)s.clusters << s.cl_log2) * (s.threads / 32) * kBfsChunk;
}

rr_status launch_bfs(BfsArgs g, const BfsShape &s, cudaStream_t st, int dtype_code) {
    g.cl_log2 = s.cl_log2;
    g.bm_words = s.bm_words;
    g.fcap = s.fcap;
    const int cpl = (g.s.row_chunks + 31) / 32;
    switch (dtype_code) {
        case DT_U8: return launch_bfs_u8(g, s, st);
        case DT_I8: return launch_bfs_i8(g, s, st);
        case DT_F32: return cpl <= 2 ? launch_bfs_f32(g, s, st) : launch_bfs_f32_wide(g, s, st);
    }
    set_error("greedy phase: unsupported element type %d", dtype_code);
    return RR_EINVAL;
}

}  // namespace rr
