// k_brute_tc.cu -- exact range search by exhaustive scan (Def. 2.1) of 8-bit
// indexes on the tensor cores.
//
// All distances of a query tile to a point tile are one matrix product: with
// every byte shifted to [-128, 127] (exact in fp16; a shift of both sides leaves
// squared L2 unchanged, and the inner product is corrected by the vectors'
// sums), the products and every partial sum are integers of magnitude at most
// 512 * 2^14 = 2^23, so the fp32 accumulators hold them exactly and the results
// equal the integer ones.  tcgen05.mma kind::f16, M = 128 queries x N points.
//
// One CTA keeps a tile of 128 queries in shared memory (fp16, K-major, 128-byte
// swizzle) and streams point tiles: sixteen producer warps load the bytes,
// convert them (a byte permute and a half2 subtract per two values) and take
// the points' norms; one thread issues the MMAs; four warps for each of the two
// accumulators read them from TMEM (a query per thread), keep the largest of
// dot - norm / 2 over 32 columns and look closer only where it reaches the
// query's threshold, so the usual column costs an add and a max.  Point stages
// and accumulators are double buffered.  The CTAs of all query tiles walk the
// same points side by side, so HBM is read about once.
//
// One pass: a match is appended to the item list as (query, key), counted in a
// register of the thread that owns the query; the output's bin sort takes the
// list.  The former form computed every distance twice with dp4a (count, then
// fill): 1,000 queries x 2*10^6 x 256 bytes, 31.6 -> 3.7 ms (GB300).  Bound: the
// producers' and the epilogue's instructions; the tensor pipe is busy a tenth of
// the time.
#include <cuda_fp16.h>

#include <algorithm>

#include "rr_common.cuh"

namespace rr {

namespace {

constexpr int kM = 128;                    // queries per tile
constexpr int kEpilogue = 256;             // two groups of four warps, one an accumulator
constexpr int kProducers = 512;
constexpr int kThreads = kEpilogue + kProducers + 32;  // and the MMA issuer
constexpr int kWaits = 1 << 20;            // tries of a wait before it gives up (about a second)
constexpr int kNormRing = 4;               // tiles whose norms are kept (an accumulator may be read while two more tiles load)

__device__ __forceinline__ uint32_t saddr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *b, uint32_t n) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(saddr(b)), "r"(n) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(b)) : "memory");
}
// one try, suspended for a microsecond at most
__device__ __forceinline__ bool mbar_try(uint64_t *b, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 1000;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok) : "r"(saddr(b)), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded waits: false when `tries` ran out or another role has given up.  A whole warp waits and votes on every
// try, so that all its lanes leave together, one way or the other: what follows (tcgen05.ld.sync.aligned, full-mask
// votes) needs the whole warp.  A lane whose try succeeded may try again: the barrier cannot complete two phases
// further without this warp's own arrival.
__device__ __forceinline__ bool mbar_wait_warp(uint64_t *b, uint32_t parity, volatile int *stop, int tries) {
    for (int i = 0; i < tries; i++) {
        if (__all_sync(0xffffffffu, mbar_try(b, parity))) return true;
        if (__any_sync(0xffffffffu, *stop != 0)) return false;
    }
    *stop = 1;
    return false;
}
// the same for a single thread
__device__ __forceinline__ bool mbar_wait_one(uint64_t *b, uint32_t parity, volatile int *stop, int tries) {
    for (int i = 0; i < tries; i++) {
        if (mbar_try(b, parity)) return true;
        if (*stop) return false;
    }
    *stop = 1;
    return false;
}

// shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups 1,024 bytes apart
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
    return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

__device__ __forceinline__ void mma_f16(uint32_t d, uint64_t ad, uint64_t bd, uint32_t idesc, bool acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d), "l"(ad), "l"(bd), "r"(idesc),
        "r"((uint32_t)acc)
        : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t *b) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(saddr(b))
                 : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t ad, uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, "
        "[%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
          "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
          "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(ad));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ uint32_t tmem_ld1(uint32_t ad) {
    uint32_t v;
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(v) : "r"(ad));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    return v;
}

struct TcArgs {
    SearchArgs a;
    int32_t n_tile;      // N: points per tile
    int32_t kpad;        // K: bytes of a row rounded up to 64
    int32_t per_group;   // CTAs per query tile
    int64_t tiles;       // point tiles
    int32_t *counts;     // per query, zero at the start
    uint32_t *lo_dk;     // per query: smallest distance key (all ones at the start)
    uint64_t *item_key;
    int32_t *item_slot;
    int64_t cap;
    unsigned long long *tail;
    int32_t wait_tries;  // tries of a wait before it gives up
};

// 16 stored bytes -> 16 fp16 values of [-128, 127], written as chunks 2c and 2c + 1 of the row; adds the row's
// sum and sum of squares
template <bool SIGNED>
__device__ __forceinline__ void convert16(const uint4 &v, uint4 &h0, uint4 &h1, int &sq, int &sum) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    uint32_t h[8];
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const uint32_t ub = SIGNED ? w[i] ^ 0x80808080u : w[i], sb = w[i] ^ (SIGNED ? 0u : 0x80808080u);
        sq = __dp4a((int)sb, (int)sb, sq);
        sum = __dp4a((int)sb, 0x01010101, sum);
        // fp16 0x64XX = 1024 + XX
        const uint32_t lo = __byte_perm(ub, 0x64646464u, 0x4140), hi = __byte_perm(ub, 0x64646464u, 0x4342);
        const __half2 off = __half2half2(__ushort_as_half(0x6480));  // 1152
        const __half2 a = __hsub2(*reinterpret_cast<const __half2 *>(&lo), off);
        const __half2 b = __hsub2(*reinterpret_cast<const __half2 *>(&hi), off);
        h[2 * i] = *reinterpret_cast<const uint32_t *>(&a);
        h[2 * i + 1] = *reinterpret_cast<const uint32_t *>(&b);
    }
    h0 = make_uint4(h[0], h[1], h[2], h[3]);
    h1 = make_uint4(h[4], h[5], h[6], h[7]);
}

// the two 16-byte chunks of stored chunk c (32 bytes of fp16) of row r in an operand tile of `rows` rows
__device__ __forceinline__ void put_chunk(uint8_t *tile, int rows, int r, int c, const uint4 &h0, const uint4 &h1) {
    uint8_t *row = tile + (size_t)(c >> 2) * rows * 128 + (size_t)r * 128;  // 64 values (4 stored chunks) a K block
    const int j = (c & 3) * 2;
    *reinterpret_cast<uint4 *>(row + ((j ^ (r & 7)) << 4)) = h0;
    *reinterpret_cast<uint4 *>(row + (((j + 1) ^ (r & 7)) << 4)) = h1;
}

// What a vector adds to the comparison, given its sum of squares and sum over the D stored bytes:
//   L2: norm2;  IP of uint8: sum (q+128)(x+128) = dot + 128 (sum q + sum x) + 128^2 D;  IP of int8: nothing
template <bool SIGNED>
__device__ __forceinline__ int side_term(int metric, int sq, int sum) {
    return metric == MET_L2 ? sq : (SIGNED ? 0 : 128 * sum);
}

template <bool SIGNED>
__global__ void __launch_bounds__(kThreads, 1) brute_tc_kernel(TcArgs g) {
    extern __shared__ uint8_t smem_dyn[];
    __shared__ __align__(8) uint64_t full[2], empty[2], tfull[2], tempty[2];
    __shared__ uint32_t tmem_base;
    __shared__ int stop_flag;
    __shared__ int qside[kM];
    __shared__ __align__(16) int xside[kNormRing][256];
    __shared__ __align__(16) float xhalf[kNormRing][256];
    const SearchArgs &a = g.a;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int N = g.n_tile, K = g.kpad, kch = K / 16;
    uint8_t *At = reinterpret_cast<uint8_t *>(((uintptr_t)smem_dyn + 1023) & ~(uintptr_t)1023);
    uint8_t *Bt = At + (size_t)kM * K * 2;
    const size_t bstage = (size_t)N * K * 2;
    volatile int *stop = &stop_flag;
    const int64_t q0 = (int64_t)(blockIdx.x / g.per_group) * kM;
    const int64_t t0 = blockIdx.x % g.per_group;
    const int nqt = (int)min((int64_t)kM, a.nq - q0);
    const int ncols = N * 2 < 32 ? 32 : N * 2;

    if (tid == 0) {
        stop_flag = 0;
        for (int s = 0; s < 2; s++) {
            mbar_init(&full[s], kProducers);
            mbar_init(&empty[s], 1);
            mbar_init(&tfull[s], 2);  // the MMAs' completion, and the issuer (carries the producers' norms)
            mbar_init(&tempty[s], 128);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();  // the .sync.aligned instructions want the whole warp
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(&tmem_base)),
                     "r"(ncols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // lane groups: a row's stored chunks over lg lanes
    int lg = 4;
    while (lg < kch) lg <<= 1;
    const int sub = lane & (lg - 1), rows_w = 32 / lg, rsub = lane / lg;
    // the query tile
    for (int r0 = warp * rows_w; r0 < kM; r0 += (kThreads / 32) * rows_w) {
        const int r = r0 + rsub;
        uint4 h0 = make_uint4(0, 0, 0, 0), h1 = h0;
        int sq = 0, sum = 0;
        if (r < nqt && sub < a.row_chunks)
            convert16<SIGNED>(ldg16(a.queries + (size_t)(q0 + r) * a.row_stride + (size_t)sub * 16), h0, h1, sq, sum);
        if (r < kM && sub < kch) put_chunk(At, kM, r, sub, h0, h1);
        for (int o = lg >> 1; o > 0; o >>= 1) {
            sq += __shfl_xor_sync(0xffffffffu, sq, o);
            sum += __shfl_xor_sync(0xffffffffu, sum, o);
        }
        if (sub == 0 && r < kM) qside[r] = side_term<SIGNED>(a.metric, sq, sum);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base;

    if (warp < kEpilogue / 32) {
        // epilogue: thread = query; group warp / 4 takes the tiles of its accumulator
        const int s = warp >> 2, row = tid & (kM - 1);
        const bool live = row < nqt;
        const int64_t qi = q0 + row;
        const uint32_t rk = live ? a.rkey[qi] : 0u;
        const bool l2 = a.metric == MET_L2;
        const int qs = qside[row];
        const int bias = l2 || SIGNED ? 0 : 16384 * a.row_stride;
        // a point is looked at when dot - xh >= thr; L2: 2 dot - xn >= qn - r, IP: dot + xs >= -r - qs - bias.
        // Everything is an integer below 2^25 but r, so 2 plus a rounding of the threshold covers the fp32 error.
        const double r = (double)dval_i32(rk);
        const double t = l2 ? 0.5 * ((double)qs - r) : -r - (double)qs - (double)bias;
        const float thr = live ? (float)(t - 2.0 - fabs(t) * 1e-6) : __int_as_float(0x7f800000);
        const uint32_t acc = tmem + (uint32_t)(s * N) + ((uint32_t)((warp & 3) * 32) << 16);
        int cnt = 0;
        uint32_t lo = 0xFFFFFFFFu;
        int it = s;
        for (int64_t tile = t0 + (int64_t)s * g.per_group; tile < g.tiles; tile += 2 * (int64_t)g.per_group, it += 2) {
            const int ring = it % kNormRing;
            if (!mbar_wait_warp(&tfull[s], (it >> 1) & 1, stop, g.wait_tries)) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int64_t p0 = tile * N;
            for (int c0 = 0; c0 < N; c0 += 32) {
                uint32_t v[32];
                tmem_ld32(acc + (uint32_t)c0, v);
                float m = -__int_as_float(0x7f800000);
#pragma unroll
                for (int j = 0; j < 32; j += 4) {
                    const float4 x = *reinterpret_cast<const float4 *>(&xhalf[ring][c0 + j]);
                    m = fmaxf(m, fmaxf(fmaxf(__uint_as_float(v[j]) - x.x, __uint_as_float(v[j + 1]) - x.y),
                                       fmaxf(__uint_as_float(v[j + 2]) - x.z, __uint_as_float(v[j + 3]) - x.w)));
                }
                if (!__any_sync(0xffffffffu, m >= thr)) continue;
                uint32_t cols = 0;
#pragma unroll
                for (int j = 0; j < 32; j++) cols |= __uint_as_float(v[j]) - xhalf[ring][c0 + j] >= thr ? 1u << j : 0u;
                for (cols = __reduce_or_sync(0xffffffffu, cols); cols; cols &= cols - 1) {
                    const int j = c0 + __ffs(cols) - 1;
                    const int64_t p = p0 + j;
                    const int dot = (int)__uint_as_float(tmem_ld1(acc + (uint32_t)j)), xs = xside[ring][j];
                    const int dist = l2 ? qs + xs - 2 * dot : -(dot + qs + xs + bias);
                    const uint32_t dk = dkey_i32(dist);
                    const bool in = live && p < a.n && dk <= rk;
                    const unsigned msk = __ballot_sync(0xffffffffu, in);
                    if (!msk) continue;
                    unsigned long long b0 = 0;
                    if (lane == 0) b0 = atomicAdd(g.tail, (unsigned long long)__popc(msk));
                    b0 = __shfl_sync(0xffffffffu, b0, 0);
                    if (in) {
                        const int64_t at = (int64_t)b0 + __popc(msk & lanemask_lt());
                        if (at < g.cap) {
                            g.item_key[at] = make_key(dk, a.ext ? __ldg(a.ext + p) : (uint32_t)p);
                            g.item_slot[at] = (int32_t)qi;
                        }
                        cnt++;
                        lo = min(lo, dk);
                    }
                    __syncwarp();  // before the next load from TMEM
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            mbar_arrive(&tempty[s]);
        }
        if (live && cnt > 0) {
            atomicAdd(g.counts + qi, cnt);
            atomicMin(g.lo_dk + qi, lo);
        }
    } else if (warp < (kEpilogue + kProducers) / 32) {
        // A thread loads up to U = 4 chunks of a tile (2,048 lane slots a tile at most); the next tile's are in flight
        // while the stage is waited for.
        const int pw = warp - kEpilogue / 32;
        constexpr int U = 4;
        const int step = (kProducers / 32) * rows_w;
        uint4 v[U];
        auto load = [&](int64_t tile) {
#pragma unroll
            for (int u = 0; u < U; u++) {
                const int r = pw * rows_w + u * step + rsub;
                const int64_t p = tile * N + r;
                v[u] = tile < g.tiles && r < N && p < a.n && sub < a.row_chunks
                           ? ldg16(a.vec + (size_t)p * a.row_stride + (size_t)sub * 16) : make_uint4(0, 0, 0, 0);
            }
        };
        load(t0);
        int it = 0;
        for (int64_t tile = t0; tile < g.tiles; tile += g.per_group, it++) {
            const int s = it & 1, ring = it % kNormRing;
            if (it >= 2 && !mbar_wait_warp(&empty[s], ((it >> 1) - 1) & 1, stop, g.wait_tries)) break;
            uint8_t *B = Bt + s * bstage;
#pragma unroll
            for (int u = 0; u < U; u++) {
                if (pw * rows_w + u * step >= N) break;  // warp-uniform
                const int r = pw * rows_w + u * step + rsub;
                uint4 h0 = make_uint4(0, 0, 0, 0), h1 = h0;
                int sq = 0, sum = 0;
                if (sub < a.row_chunks) convert16<SIGNED>(v[u], h0, h1, sq, sum);
                if (sub < kch) put_chunk(B, N, r, sub, h0, h1);
                for (int o = lg >> 1; o > 0; o >>= 1) {
                    sq += __shfl_xor_sync(0xffffffffu, sq, o);
                    sum += __shfl_xor_sync(0xffffffffu, sum, o);
                }
                if (sub == 0) {
                    const int x = side_term<SIGNED>(a.metric, sq, sum);
                    xside[ring][r] = x;
                    xhalf[ring][r] = a.metric == MET_L2 ? 0.5f * (float)x : -(float)x;
                }
            }
            load(tile + g.per_group);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbar_arrive(&full[s]);
        }
    } else if (lane == 0) {
        // the MMA issuer.  Instruction descriptor: D fp32, A and B fp16, both K-major, N / 8, M / 16
        const uint32_t idesc = (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(kM >> 4) << 24);
        const uint32_t abase = saddr(At), bbase = saddr(Bt);
        int it = 0;
        for (int64_t tile = t0; tile < g.tiles; tile += g.per_group, it++) {
            const int s = it & 1;
            if (!mbar_wait_one(&full[s], (it >> 1) & 1, stop, g.wait_tries)) break;
            if (it >= 2 && !mbar_wait_one(&tempty[s], ((it >> 1) - 1) & 1, stop, g.wait_tries)) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            for (int k = 0; k < K / 16; k++) {  // 16 values (32 bytes) a step, 64 a swizzled block
                const uint32_t ka = abase + (uint32_t)(k >> 2) * kM * 128 + (k & 3) * 32;
                const uint32_t kb = bbase + (uint32_t)(s * bstage) + (uint32_t)(k >> 2) * N * 128 + (k & 3) * 32;
                mma_f16(tmem + (uint32_t)(s * N), smem_desc(ka), smem_desc(kb), idesc, k > 0);
            }
            mma_commit(&empty[s]);
            mma_commit(&tfull[s]);
            mbar_arrive(&tfull[s]);
        }
        // every MMA has read its operands and written its accumulators, and every commit has arrived on its barrier,
        // before the CTA goes on (also when an epilogue group left early)
        for (int t = it > 2 ? it - 2 : 0; t < it; t++)
            for (int i = 0; i < kWaits && !(mbar_try(&empty[t & 1], (t >> 1) & 1) && mbar_try(&tfull[t & 1], (t >> 1) & 1)); i++) {}
    }
    __syncwarp();
    __syncthreads();
    if (tid == 0 && stop_flag) atomicExch(a.error, 8);
    __syncwarp();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
}

}  // namespace

bool brute_tc(int dtype_code) { return dtype_code == DT_U8 || dtype_code == DT_I8; }

rr_status launch_brute_tc(const SearchArgs &a, int32_t *counts, uint32_t *lo_dk, uint64_t *item_key, int32_t *item_slot,
                          int64_t cap, unsigned long long *tail, cudaStream_t st, int dtype_code) {
    if (a.nq == 0 || a.n == 0) return RR_OK;
    TcArgs g;
    g.a = a;
    g.kpad = (a.row_stride + 63) / 64 * 64;
    if (g.kpad > 512) {
        set_error("brute force: 8-bit rows above 512 bytes");
        return RR_EINVAL;
    }
    // points per tile: two stages beside the query tile in 227 KB, at most 256
    const int k = g.kpad;
    g.n_tile = k <= 128 ? 256 : (k <= 256 ? 128 : (k <= 384 ? 64 : 32));
    g.tiles = (a.n + g.n_tile - 1) / g.n_tile;
    const int64_t groups = (a.nq + kM - 1) / kM;
    g.per_group = (int32_t)std::min<int64_t>(g.tiles, std::max<int64_t>(1, 152 / groups));
    g.counts = counts;
    g.lo_dk = lo_dk;
    g.item_key = item_key;
    g.item_slot = item_slot;
    g.cap = cap;
    g.tail = tail;
    g.wait_tries = brute_wait_tries(kWaits);
    const size_t smem = 1024 + (size_t)kM * k * 2 + 2 * (size_t)g.n_tile * k * 2;
    auto kern = dtype_code == DT_U8 ? brute_tc_kernel<false> : brute_tc_kernel<true>;
    if (rr_status e = allow_smem((const void *)kern, smem)) return e;
    kern<<<(unsigned)(groups * g.per_group), kThreads, smem, st>>>(g);
    RR_CUDA(cudaGetLastError());
    note_launch();
    return RR_OK;
}

}  // namespace rr
