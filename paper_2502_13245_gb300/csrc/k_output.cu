// k_output.cu -- assembly of the per-query results into one CSR (the output
// of Alg. 6 / Alg. 3 for the whole batch): count -> exclusive scan -> copy or
// scatter -> per-query sort by (distance, id) -> decode keys into ids and
// distances.
//
// Two sorts: a few results go straight to their segments and a CTA sorts each
// (scatter_items + sort_segments); many results are first distributed into
// distance bins of about 16 keys and a warp sorts each bin in registers
// (launch_bin_sort).
#include <algorithm>

#include "rr_common.cuh"

namespace rr {

namespace {

// Exclusive scan of int32 counts into int64 offsets[0..n], one CTA, chunked.
__global__ void __launch_bounds__(1024) scan_kernel(const int32_t *counts, int64_t n, int64_t *offsets) {
    __shared__ int64_t wsum[32];
    __shared__ int64_t carry;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    if (t == 0) carry = 0;
    __syncthreads();
    for (int64_t base = 0; base < n; base += 1024) {
        int64_t i = base + t;
        int64_t v = i < n ? (int64_t)counts[i] : 0;
        int64_t x = v;
        for (int o = 1; o < 32; o <<= 1) {
            int64_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[w] = x;
        __syncthreads();
        if (w == 0) {
            int64_t s = wsum[lane];
            for (int o = 1; o < 32; o <<= 1) {
                int64_t y = __shfl_up_sync(0xffffffffu, s, o);
                if (lane >= o) s += y;
            }
            wsum[lane] = s;  // inclusive prefix of warp sums
        }
        __syncthreads();
        int64_t incl = x + (w > 0 ? wsum[w - 1] : 0) + carry;
        if (i < n) offsets[i] = incl - v;
        __syncthreads();
        if (t == 1023) carry = incl;
        __syncthreads();
    }
    if (t == 0) offsets[n] = carry;
}

__device__ __forceinline__ void decode_to(const OutArgs &o, int64_t pos, uint64_t k) {
    if (pos < 0 || pos >= o.total) {  // never write outside the result arrays
        atomicExch(o.error, 4);
        return;
    }
    const uint32_t id = key_id(k);
    o.ids[pos] = o.ext ? __ldg(o.ext + id) : id;
    uint32_t dk = key_dk(k);
    if (o.dist_is_float) reinterpret_cast<float *>(o.dists)[pos] = dval_f32(dk);
    else reinterpret_cast<int32_t *>(o.dists)[pos] = dval_i32(dk);
}

// Warp per listed slot: copy `count[slot]` sorted keys from keys[slot*stride]
// to the CSR range of query qlist[slot] (qlist == nullptr: slot = query, and
// queries flagged RR_FLAG_PHASE2 are skipped -- their results come later).
__global__ void copy_slots_kernel(OutArgs o, const uint64_t *keys, int64_t stride, const int32_t *count,
                                  const int32_t *qlist, int32_t nlist) {
    const int lane = lane_id();
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t s = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); s < nlist; s += nw) {
        int64_t q = qlist ? qlist[s] : s;
        if (!qlist && (o.flags[q] & RR_FLAG_PHASE2)) continue;
        int32_t c = count[s];
        int64_t off = o.offsets[q];
        const uint64_t *src = keys + (size_t)s * stride;
        for (int i = lane; i < c; i += 32) decode_to(o, off + i, src[i]);
    }
}

// Items to the CSR segments of their queries (unsorted within a segment).  Items come in runs of one
// slot, so the first lane of each run in a warp reserves the run's positions with one atomic.
__global__ void scatter_items_kernel(OutArgs o, const uint64_t *item_key, const int32_t *item_slot, int64_t nitems,
                                     const int32_t *qlist, int32_t *cursor, uint64_t *tmp) {
    const int lane = lane_id();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) & ~(int64_t)31; base < nitems; base += stride) {
        const int64_t t = base + lane;
        const int32_t s = t < nitems ? item_slot[t] : -1;
        const bool ok = s >= 0;
        const int32_t prev = __shfl_up_sync(0xffffffffu, s, 1);
        const bool head = ok && (lane == 0 || prev != s);
        const unsigned hm = __ballot_sync(0xffffffffu, head);
        int32_t r0 = 0;
        // a run ends at the next lane of another slot, or of none
        const unsigned brk = __ballot_sync(0xffffffffu, lane == 0 || prev != s);
        if (head) {
            const unsigned later = brk & ~((2u << lane) - 1u);
            r0 = atomicAdd(cursor + s, (later ? __ffs(later) - 1 : 32) - lane);
        }
        // the head of this lane's run: the last head at or before the lane (lane 0 is one when ok)
        const unsigned upto = hm & ((2u << lane) - 1u);
        const int h = upto ? 31 - __clz(upto) : 0;
        r0 = __shfl_sync(0xffffffffu, r0, h);
        if (!ok) continue;
        const int64_t q = qlist ? qlist[s] : s;
        const int64_t pos = o.offsets[q] + r0 + (lane - h);
        if (pos < 0 || pos >= o.offsets[q + 1]) {
            atomicExch(o.error, 4);
            continue;
        }
        tmp[pos] = item_key[t];
    }
}

// Bitonic sort with "flip" first stages, so every compare puts the smaller key
// at the lower index and a virtual +inf padding past m never moves.  The
// stages whose pairs lie inside one 64-key region (every stage of the levels
// k <= 64, and the j <= 32 stages of every later level) run in registers: a
// warp holds a region as keys r + lane and r + 32 + lane and exchanges them by
// shuffles, so only the j >= 64 stages go through memory with a block barrier.

// one stage on a warp's 64-key region (x = key lane, y = key 32 + lane)
__device__ __forceinline__ void region_stage(uint64_t &x, uint64_t &y, int lane, int k, int j) {
    const bool flip = j == (k >> 1);
    if (j == 32) {
        if (flip) {  // k = 64: key lane pairs with key 63 - lane, the y of lane 31 - lane
            const uint64_t oy = __shfl_xor_sync(0xffffffffu, y, 31);
            const uint64_t ox = __shfl_xor_sync(0xffffffffu, x, 31);
            x = oy < x ? oy : x;
            y = ox > y ? ox : y;
        } else {
            const uint64_t lo = x < y ? x : y, hi = x < y ? y : x;
            x = lo;
            y = hi;
        }
    } else {
        const int partner = flip ? k - 1 : j;  // pair (t, t ^ (k-1)) or (t, t + j), both within 32 keys
        const uint64_t ox = __shfl_xor_sync(0xffffffffu, x, partner);
        const uint64_t oy = __shfl_xor_sync(0xffffffffu, y, partner);
        const bool upper = (lane & j) != 0;  // the higher index of the pair keeps the larger key
        x = upper ? (ox > x ? ox : x) : (ox < x ? ox : x);
        y = upper ? (oy > y ? oy : y) : (oy < y ? oy : y);
    }
}

// stages (k, j) for j from j_hi down to 1 on every 64-key region (keys past m read as +inf, not stored)
__device__ __forceinline__ void region_pass(uint64_t *a, int m, int P, int k, int j_hi, bool levels_upto_64) {
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int r = threadIdx.x >> 5; r < (P >> 6); r += nw) {
        const int i0 = (r << 6) + lane, i1 = i0 + 32;
        uint64_t x = i0 < m ? a[i0] : ~0ull, y = i1 < m ? a[i1] : ~0ull;
        if (levels_upto_64) {
#pragma unroll
            for (int kk = 2; kk <= 64; kk <<= 1)
#pragma unroll
                for (int j = kk >> 1; j > 0; j >>= 1) region_stage(x, y, lane, kk, j);
        } else {
#pragma unroll
            for (int j = 32; j > 0; j >>= 1)
                if (j <= j_hi) region_stage(x, y, lane, k, j);
        }
        if (i0 < m) a[i0] = x;
        if (i1 < m) a[i1] = y;
    }
}

__device__ void bitonic_sort_smem(uint64_t *a, int m) {
    int P = 64;
    while (P < m) P <<= 1;
    region_pass(a, m, P, 64, 32, true);
    __syncthreads();
    for (int k = 128; k <= P; k <<= 1) {
        for (int j = k >> 1; j >= 64; j >>= 1) {
            const int lj = __ffs(j) - 1;  // j and k are powers of two: shifts and masks, no divisions
            for (int i = threadIdx.x; i < P / 2; i += blockDim.x) {
                // i-th compare pair of this stage
                const int off = i & (j - 1);
                const int lo = ((i >> lj) << (lj + 1)) + off;
                // flip stage: pair (x, x ^ (k-1)) inside each k-block; otherwise (x, x + j)
                const int hi = (j == (k >> 1)) ? lo - off + (k - 1 - off) : lo + j;
                if (hi < m) {
                    uint64_t x = a[lo], y = a[hi];
                    if (y < x) { a[lo] = y; a[hi] = x; }
                }
            }
            __syncthreads();
        }
        region_pass(a, m, P, k, 32, false);
        __syncthreads();
    }
}

// CTA per listed query: sort its CSR segment of tmp keys and decode it.
// Segments up to smem_cap keys are sorted in shared memory, longer ones in
// place in global memory with the same network.
__global__ void __launch_bounds__(1024) sort_segments_kernel(OutArgs o, uint64_t *tmp, const int32_t *qlist,
                                                             int32_t nlist, int smem_cap) {
    extern __shared__ __align__(16) uint8_t smem_raw[];
    uint64_t *sk = reinterpret_cast<uint64_t *>(smem_raw);
    for (int32_t s = blockIdx.x; s < nlist; s += gridDim.x) {
        int64_t q = qlist ? qlist[s] : s;
        int64_t off = o.offsets[q];
        int m = (int)(o.offsets[q + 1] - off);
        if (m <= 0) continue;
        uint64_t *seg = tmp + off;
        uint64_t *a = seg;
        if (m <= smem_cap) {
            for (int i = threadIdx.x; i < m; i += blockDim.x) sk[i] = seg[i];
            __syncthreads();
            a = sk;
        }
        bitonic_sort_smem(a, m);
        for (int i = threadIdx.x; i < m; i += blockDim.x) decode_to(o, off + i, a[i]);
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------------------------
// Bin sort.  A segment's keys are distributed into nb = count / 16 bins of equal distance width
// between its closest beam result and its radius, and each bin is sorted on its own: the bins are in
// order, so the sorted bins side by side are the sorted segment.  Every key is read and written a
// constant number of times, whatever the segment's length, where the bitonic sort of one CTA per
// segment did log^2 passes, in global memory above 29,056 keys.  Measured (GB300, 2*10^6 x 256, whole search):
// 2,048 queries with 36.0 M results, up to 215,000 each, 35.0 -> 21.7 ms; 20,000 queries with 5.6 M results
// 8.49 -> 7.43 ms.  Bound: the returning atomics of the rank pass and the random 8-byte writes of the scatter.
// ---------------------------------------------------------------------------------------------
constexpr int kBinKeys = 16;       // mean keys per bin; a peaked distance distribution triples it locally
constexpr int kWarpBin = 256;      // larger bins (many equal distances) go to a CTA sort

__device__ __forceinline__ uint32_t bin_of(const SlotBins &b, uint32_t dk) {
    return b.base + __umulhi(dk > b.lo ? dk - b.lo : 0u, b.scale);
}

// bins of each slot: scale = floor((nb * 2^32 - 1) / (range + 1)) <= 2^32 - 1 keeps the bin below nb and
// non-decreasing in the distance
__global__ void bin_setup_kernel(BinSortArgs a) {
    for (int32_t s = blockIdx.x * blockDim.x + threadIdx.x; s < a.nslots; s += gridDim.x * blockDim.x) {
        const int64_t q = a.qlist ? a.qlist[s] : s;
        const int32_t c = a.slot_count[s];
        SlotBins b{0, 0, 0, 0};
        if (c > 0) {
            const uint32_t rk = a.rkey[q];
            b.lo = min(a.lo_keys ? key_dk(a.lo_keys[(size_t)q * a.lo_stride]) : a.lo_dk[s], rk);
            const uint64_t range = (uint64_t)(rk - b.lo) + 1;
            uint64_t nb = max(1, c / kBinKeys);
            if (nb > range) nb = range;
            b.nb = (uint32_t)nb;
            b.scale = nb == 1 ? 0u : (uint32_t)(((nb << 32) - 1) / range);
            b.base = atomicAdd(a.ctr, b.nb);
        }
        a.info[s] = b;
    }
}

// an item's place within its bin (arbitrary: the bin is sorted later)
__global__ void __launch_bounds__(256) bin_rank_kernel(BinSortArgs a) {
    constexpr int U = 4;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t0 < a.nitems; t0 += stride * U) {
        int32_t s[U];
        uint32_t dk[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int64_t t = t0 + u * stride;
            s[u] = t < a.nitems ? a.item_slot[t] : -1;
            dk[u] = t < a.nitems ? key_dk(a.item_key[t]) : 0u;
        }
        uint32_t r[U];
#pragma unroll
        for (int u = 0; u < U; u++)
            if (s[u] >= 0) r[u] = atomicAdd(a.bin_cnt + bin_of(a.info[s[u]], dk[u]), 1u);
#pragma unroll
        for (int u = 0; u < U; u++)
            if (s[u] >= 0) a.rank[t0 + u * stride] = r[u];
    }
}

// CSR position of every bin: exclusive scan of the counts of each slot, from its segment's start.  A warp
// per slot of up to 512 bins, then the CTA for each longer one.
__global__ void __launch_bounds__(256) bin_scan_kernel(BinSortArgs a) {
    __shared__ uint32_t wsum[8];
    const int lane = lane_id(), w = threadIdx.x >> 5;
    const int64_t nw = (int64_t)gridDim.x * 8;
    for (int64_t s = (int64_t)blockIdx.x * 8 + w; s < a.nslots; s += nw) {
        const SlotBins b = a.info[s];
        if (b.nb == 0 || b.nb > 512) continue;
        int64_t at = a.o.offsets[a.qlist ? a.qlist[s] : s];
        for (uint32_t i0 = 0; i0 < b.nb; i0 += 32) {
            const uint32_t i = i0 + lane, v = i < b.nb ? a.bin_cnt[b.base + i] : 0u;
            uint32_t x = v;
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            if (i < b.nb) a.bin_start[b.base + i] = at + x - v;
            at += __shfl_sync(0xffffffffu, x, 31);
        }
    }
    for (int32_t s = blockIdx.x; s < a.nslots; s += gridDim.x) {
        const SlotBins b = a.info[s];
        if (b.nb <= 512) continue;  // uniform over the CTA
        int64_t at = a.o.offsets[a.qlist ? a.qlist[s] : s];
        for (uint32_t i0 = 0; i0 < b.nb; i0 += 1024) {
            const uint32_t i = i0 + threadIdx.x * 4;
            uint32_t v[4], sum = 0;
#pragma unroll
            for (int k = 0; k < 4; k++) {
                v[k] = i + k < b.nb ? a.bin_cnt[b.base + i + k] : 0u;
                sum += v[k];
            }
            uint32_t x = sum;
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            if (lane == 31) wsum[w] = x;
            __syncthreads();
            uint32_t before = 0, total = 0;
#pragma unroll
            for (int k = 0; k < 8; k++) {
                if (k < w) before += wsum[k];
                total += wsum[k];
            }
            int64_t p = at + before + x - sum;
#pragma unroll
            for (int k = 0; k < 4; k++) {
                if (i + k < b.nb) a.bin_start[b.base + i + k] = p;
                p += v[k];
            }
            at += total;
            __syncthreads();
        }
    }
}

__global__ void __launch_bounds__(256) bin_scatter_kernel(BinSortArgs a) {
    constexpr int U = 4;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t0 < a.nitems; t0 += stride * U) {
        int32_t s[U];
        uint64_t k[U];
        int64_t pos[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int64_t t = t0 + u * stride;
            s[u] = t < a.nitems ? a.item_slot[t] : -1;
            k[u] = t < a.nitems ? a.item_key[t] : 0ull;
            pos[u] = s[u] >= 0 ? (int64_t)a.rank[t] : 0;
        }
#pragma unroll
        for (int u = 0; u < U; u++)
            if (s[u] >= 0) pos[u] += a.bin_start[bin_of(a.info[s[u]], key_dk(k[u]))];
#pragma unroll
        for (int u = 0; u < U; u++)
            if (s[u] >= 0) {
                if (pos[u] < a.o.total) a.tmp[pos[u]] = k[u];
                else atomicExch(a.o.error, 4);  // counts and items disagree: cannot happen
            }
    }
}

// one stage of a 32-key network, a key per lane (flip: the first stage of a level)
__device__ __forceinline__ void lane_stage(uint64_t &x, int lane, int k, int j) {
    const uint64_t o = __shfl_xor_sync(0xffffffffu, x, j == (k >> 1) ? k - 1 : j);
    const bool upper = (lane & j) != 0;
    x = upper ? (o > x ? o : x) : (o < x ? o : x);
}

// a warp per bin: up to 64 keys in registers, up to kWarpBin in shared memory, the rest listed
__global__ void __launch_bounds__(256) bin_sort_kernel(BinSortArgs a) {
    __shared__ uint64_t sk[8][kWarpBin];
    const int lane = lane_id(), w = threadIdx.x >> 5;
    const uint32_t nbins = a.ctr[0], nw = gridDim.x * 8;
    for (uint32_t i = blockIdx.x * 8 + w; i < nbins; i += nw) {
        const uint32_t c = a.bin_cnt[i];
        const int64_t p = a.bin_start[i];
        if (c == 0 || p + c > a.o.total) continue;
        if (c <= 32) {
            uint64_t x = lane < c ? a.tmp[p + lane] : kEmpty;
            for (int k = 2; k < 2 * (int)c; k <<= 1)  // levels up to the power of two that holds c keys
                for (int j = k >> 1; j > 0; j >>= 1) lane_stage(x, lane, k, j);
            if (lane < c) decode_to(a.o, p + lane, x);
        } else if (c <= 64) {
            uint64_t x = a.tmp[p + lane], y = 32 + lane < c ? a.tmp[p + 32 + lane] : kEmpty;
#pragma unroll
            for (int k = 2; k <= 64; k <<= 1)
#pragma unroll
                for (int j = k >> 1; j > 0; j >>= 1) region_stage(x, y, lane, k, j);
            decode_to(a.o, p + lane, x);
            if (32 + lane < c) decode_to(a.o, p + 32 + lane, y);
        } else if (c <= kWarpBin) {
            for (uint32_t t = lane; t < c; t += 32) sk[w][t] = a.tmp[p + t];
            __syncwarp();
            warp_sort_keys(sk[w], (int)c);
            for (uint32_t t = lane; t < c; t += 32) decode_to(a.o, p + t, sk[w][t]);
            __syncwarp();
        } else if (lane == 0) {
            a.big[atomicAdd(a.ctr + 1, 1u)] = i;
        }
    }
}

// a CTA per listed bin, in shared memory up to smem_cap keys, in place beyond
__global__ void __launch_bounds__(1024) bin_sort_big_kernel(BinSortArgs a, int smem_cap) {
    extern __shared__ __align__(16) uint8_t smem_raw[];
    uint64_t *sk = reinterpret_cast<uint64_t *>(smem_raw);
    const uint32_t n = a.ctr[1];
    for (uint32_t x = blockIdx.x; x < n; x += gridDim.x) {
        const uint32_t i = a.big[x];
        const int m = (int)a.bin_cnt[i];
        const int64_t p = a.bin_start[i];
        uint64_t *k = a.tmp + p;
        if (m <= smem_cap) {
            for (int t = threadIdx.x; t < m; t += blockDim.x) sk[t] = k[t];
            __syncthreads();
            k = sk;
        }
        bitonic_sort_smem(k, m);
        for (int t = threadIdx.x; t < m; t += blockDim.x) decode_to(a.o, p + t, k[t]);
        __syncthreads();
    }
}

size_t ru256(size_t x) { return (x + 255) & ~size_t(255); }

// what the bin sort needs beside the keys: rank per item | bins | slots | list of large bins | counters
struct BinLayout {
    size_t rank, cnt, start, info, big, ctr, end;
    BinLayout(int64_t nitems, int64_t nslots, size_t at) {
        const size_t nb = (size_t)(nitems / kBinKeys + nslots);
        rank = ru256(at);
        ctr = rank + ru256((size_t)nitems * 4);  // counters and bin counts side by side: one memset
        cnt = ctr + 256;
        start = cnt + ru256(nb * 4);
        info = start + ru256(nb * 8);
        big = info + ru256((size_t)nslots * sizeof(SlotBins));
        end = big + ru256((size_t)(nitems / kWarpBin + 1) * 4);
    }
};

}  // namespace

size_t bin_sort_end(int64_t nitems, int64_t nslots, size_t at) { return BinLayout(nitems, nslots, at).end; }

rr_status launch_bin_sort(BinSortArgs a, uint8_t *base, size_t at, cudaStream_t st) {
    if (a.nitems <= 0 || a.nslots <= 0) return RR_OK;
    const BinLayout L(a.nitems, a.nslots, at);
    a.rank = (uint32_t *)(base + L.rank);
    a.ctr = (uint32_t *)(base + L.ctr);
    a.bin_cnt = (uint32_t *)(base + L.cnt);
    a.bin_start = (int64_t *)(base + L.start);
    a.info = (SlotBins *)(base + L.info);
    a.big = (uint32_t *)(base + L.big);
    RR_CUDA(cudaMemsetAsync(base + L.ctr, 0, L.start - L.ctr, st));
    bin_setup_kernel<<<(a.nslots + 255) / 256, 256, 0, st>>>(a);
    const unsigned ib = (unsigned)std::max<int64_t>(1, std::min<int64_t>((a.nitems + 1023) / 1024, 152 * 8));
    bin_rank_kernel<<<ib, 256, 0, st>>>(a);
    const unsigned sb = (unsigned)std::min<int64_t>((a.nslots + 7) / 8, 152 * 8);
    bin_scan_kernel<<<std::max(sb, (unsigned)std::min<int64_t>(a.nitems / (kBinKeys * 512), 152 * 4)), 256, 0, st>>>(a);
    bin_scatter_kernel<<<ib, 256, 0, st>>>(a);
    const int64_t nb = a.nitems / kBinKeys + a.nslots;
    bin_sort_kernel<<<(unsigned)std::min<int64_t>((nb + 7) / 8, 152 * 8), 256, 0, st>>>(a);
    int dev = 0, optin = 0;
    RR_CUDA(cudaGetDevice(&dev));
    RR_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    const int smem_cap = std::max(4096, optin / 8);
    if (rr_status e = allow_smem((const void *)bin_sort_big_kernel, smem_cap * 8)) return e;
    bin_sort_big_kernel<<<(unsigned)std::min<int64_t>(a.nitems / kWarpBin + 1, 152), 1024, (size_t)smem_cap * 8, st>>>(
        a, smem_cap);
    RR_CUDA(cudaGetLastError());
    note_launch(6);
    return RR_OK;
}

rr_status launch_scan(const int32_t *counts, int64_t n, int64_t *offsets, cudaStream_t st) {
    scan_kernel<<<1, 1024, 0, st>>>(counts, n, offsets);
    RR_CUDA(cudaGetLastError());
    note_launch();
    return RR_OK;
}

rr_status launch_copy_slots(const OutArgs &o, const uint64_t *keys, int64_t stride, const int32_t *count,
                            const int32_t *qlist, int32_t nlist, cudaStream_t st) {
    if (nlist <= 0) return RR_OK;
    int64_t blocks = (nlist + 7) / 8;
    if (blocks > 152 * 16) blocks = 152 * 16;
    copy_slots_kernel<<<(unsigned)blocks, 256, 0, st>>>(o, keys, stride, count, qlist, nlist);
    RR_CUDA(cudaGetLastError());
    note_launch();
    return RR_OK;
}

rr_status launch_scatter_items(const OutArgs &o, const uint64_t *item_key, const int32_t *item_slot, int64_t nitems,
                               const int32_t *qlist, int32_t *cursor, uint64_t *tmp, cudaStream_t st) {
    if (nitems <= 0) return RR_OK;
    int64_t blocks = (nitems + 255) / 256;
    if (blocks > 152 * 32) blocks = 152 * 32;
    scatter_items_kernel<<<(unsigned)blocks, 256, 0, st>>>(o, item_key, item_slot, nitems, qlist, cursor, tmp);
    RR_CUDA(cudaGetLastError());
    note_launch();
    return RR_OK;
}

rr_status launch_sort_segments(const OutArgs &o, uint64_t *tmp, const int32_t *qlist, int32_t nlist, int64_t,
                               cudaStream_t st) {
    if (nlist <= 0) return RR_OK;
    // keys: the largest shared-memory block a CTA may take (227 KB), so segments of up to 29,056 results
    // are sorted on chip; longer ones in place in global memory.  (Size classes in three launches with
    // smaller blocks for short segments measured slower: each launch has its own tail.)
    int dev = 0, optin = 0;
    RR_CUDA(cudaGetDevice(&dev));
    RR_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    const int smem_cap = std::max(4096, optin / 8);
    size_t smem = (size_t)smem_cap * 8;
    if (rr_status e = allow_smem((const void *)sort_segments_kernel, smem)) return e;
    int blocks = nlist < 152 * 2 ? nlist : 152 * 2;
    sort_segments_kernel<<<blocks, 1024, smem, st>>>(o, tmp, qlist, nlist, smem_cap);
    RR_CUDA(cudaGetLastError());
    note_launch();
    return RR_OK;
}

}  // namespace rr
