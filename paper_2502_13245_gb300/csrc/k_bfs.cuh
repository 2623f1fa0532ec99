// k_bfs.cuh -- Alg. 2 GreedySearch, a cluster of CTAs per query: the whole
// breadth-first expansion of a query (see k_greedy.cu for why the order does
// not matter) runs in one kernel, its exact bitmap of seen ids in shared memory.
//
// Why: nearly all of the work is probing the seen bit of every out-neighbour of
// every result (64 probes a result, ~98% find the bit set).  As two flat passes
// over all queries the probes go to n-bit bitmaps in global memory: each is an
// L1 tag lookup and mostly an L2 sector, a warp's 32 probes take 32 of them, and
// every level costs two launches and a host round trip.  In shared memory a
// warp's probes take a few bank-conflict cycles and a level costs one barrier.
//
// Layout: a CTA holds up to ~1.7 M bits; larger indexes spread the bitmap over a
// cluster of 2 or 4 CTAs (word w in CTA w mod CL) and probe it through
// distributed shared memory.  (A pair whose CTAs each take every item and probe
// only their own half moves no probe between SMs but was slower: 1.30 -> 1.77 ms
// at 836 queries with 5.6 M results.)  Clusters are persistent and take queries
// from a device counter.  Warps are independent within a level: a warp takes an item,
// tests and sets the bits of its row (the next item's row is loading), collects
// the first-seen ids, evaluates 32 of them at a time and appends the in-range
// ones to the query's next frontier (an L2-resident list) and to its own chunk
// of the global item list, so no counter is shared between queries.
//
// The last few large queries, once the rest of the chip has run dry, are handed
// to the two-pass levels (bitmap and frontier are copied out): a CTA does ~3
// probes per clock, the flat passes ~86 over the chip.  So is a query whose
// frontier outgrows its list.
//
// Measured (GB300, greedy phase): 836 queries, 5.6 M results, 2*10^6 x 256 u8
// 2.62 -> 1.32 ms; 1,163 queries, 36.0 M results 18.3 -> 9.2 ms; 265 queries,
// 0.47 M results, 10^6 x 128 u8 0.56 -> 0.14 ms; 520 queries, 0.53 M results,
// 10^6 x 200 fp32 0.98 -> 0.52 ms.  Bound: the bitmap probes at about half of the
// issue slots; small queries by the latency of their levels.  768 threads a CTA
// (80 registers) keep the prefetched rows out of spills: 9.2 ms against 9.9 at
// 1,024 and 10.4 at 512.
#pragma once
#include "rr_common.cuh"

namespace rr {

namespace {

constexpr int kChunk = kBfsChunk;    // items a warp reserves at a time
constexpr int kCand = 32 + 128;      // first-seen ids a warp holds: a batch and a full row
constexpr int kWarpBytes = 32 * 8 + kCand * 4;
constexpr int kCtlBytes = 64;
constexpr int kHandOver = 1, kStop = 2;

struct Ctl {                         // the copies of the cluster's first CTA are used
    int32_t slot;
    int32_t bail[2];                 // kHandOver or kStop, by level parity: written during a level, read after the
                                     // barrier that ends it
    int32_t hand;                    // hand-over: the query's bitmap in global memory, or -1
    uint32_t pend;                   // and its place in the list of pending items
    uint32_t cnt[3];                 // frontier sizes of three consecutive levels
};

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ uint32_t ld_cl(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t or_cl(uint32_t addr, uint32_t bits) {
    uint32_t v;
    asm volatile("atom.shared::cluster.or.b32 %0, [%1], %2;" : "=r"(v) : "r"(addr), "r"(bits) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t add_cl(uint32_t addr, uint32_t x) {
    uint32_t v;
    asm volatile("atom.shared::cluster.add.u32 %0, [%1], %2;" : "=r"(v) : "r"(addr), "r"(x) : "memory");
    return v;
}

// CL: the bitmap is spread over a cluster of 2^cl_log2 CTAs
template <bool CL>
struct Team {
    uint32_t rank, log2;
    uint32_t bits;       // shared address of this CTA's bitmap
    uint32_t ctl0;       // cluster address of the first CTA's Ctl
    uint32_t *bm;
    Ctl *ctl;
    __device__ __forceinline__ void sync() const {
        if constexpr (CL) {
            asm volatile("barrier.cluster.arrive.release;" ::: "memory");
            asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
        } else {
            __syncthreads();
        }
    }
    // address of the word with id's bit, the word, and setting the bit (returns the word before)
    __device__ __forceinline__ uint32_t at(uint32_t id) const {
        const uint32_t w = id >> 5;
        if constexpr (CL) return map_rank(bits + ((w >> log2) << 2), w & ((1u << log2) - 1));
        else return w;
    }
    __device__ __forceinline__ uint32_t word(uint32_t ad) const {
        if constexpr (CL) return ld_cl(ad);
        else return reinterpret_cast<volatile uint32_t *>(bm)[ad];
    }
    __device__ __forceinline__ uint32_t set(uint32_t ad, uint32_t bit) const {
        if constexpr (CL) return or_cl(ad, bit);
        else return atomicOr(bm + ad, bit);
    }
    __device__ __forceinline__ uint32_t get(const void *field) const {
        if constexpr (CL) return ld_cl(ctl0 + (uint32_t)((const uint8_t *)field - (const uint8_t *)ctl));
        else return *reinterpret_cast<const volatile uint32_t *>(field);
    }
    __device__ __forceinline__ uint32_t add(uint32_t *field, uint32_t x) const {
        if constexpr (CL) return add_cl(ctl0 + (uint32_t)((uint8_t *)field - (uint8_t *)ctl), x);
        else return atomicAdd(field, x);
    }
};

// RR: words of an adjacency row per lane (1, 2 or 4); a warp takes 4 / RR items at a time, so that each lane has
// four bitmap words in flight
template <int DT, int CPL, int RR, bool CL>
__global__ void __launch_bounds__(kBfsThreads, 1) bfs_kernel(BfsArgs g) {
    extern __shared__ __align__(16) uint8_t smem_raw[];
    constexpr int IW = 4 / RR;
    constexpr int UN = CPL == 1 ? 8 : (CPL == 2 ? 4 : 2);
    const SearchArgs &a = g.s;
    const int lane = lane_id(), warp = threadIdx.x >> 5, W = blockDim.x >> 5;
    const int R = a.R, b = a.beam;
    Team<CL> T;
    T.rank = 0;
    T.log2 = g.cl_log2;
    T.bm = reinterpret_cast<uint32_t *>(smem_raw);
    uint8_t *wb = smem_raw + (size_t)g.bm_words * 4 + (size_t)warp * kWarpBytes;
    uint64_t *ckey = reinterpret_cast<uint64_t *>(wb);
    uint32_t *cid = reinterpret_cast<uint32_t *>(wb + 32 * 8);
    T.ctl = reinterpret_cast<Ctl *>(smem_raw + (size_t)g.bm_words * 4 + (size_t)W * kWarpBytes);
    T.bits = smem_addr(T.bm);
    T.ctl0 = 0;
    if constexpr (CL) {
        asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(T.rank));
        T.ctl0 = map_rank(smem_addr(T.ctl), 0);
    }
    const uint32_t gw = T.rank * W + warp, stride = (uint32_t)W << T.log2;  // this warp and the warps of the team
    uint32_t *fr = g.front + (size_t)(blockIdx.x >> T.log2) * 2 * g.fcap;
    const bool chief = T.rank == 0 && threadIdx.x == 0;
    const int32_t np2 = *g.np2;
    // the caller's cap on the results (first beams are always kept), and the end of a run that will be redone
    auto cap = [&]() { return (unsigned long long)max(g.max_results, (int64_t)np2 * b); };
    auto give_up = [&]() {
        *g.overflow = 1;
        atomicMax(g.next, np2);  // no more queries
    };
    // this warp's chunk of the item list
    int64_t cbase = 0;
    int cfill = kChunk;

    for (;;) {
        if (chief) {
            const unsigned long long found = *(volatile unsigned long long *)g.results;  // both in flight together
            const int32_t next = atomicAdd(g.next, 1);
            T.ctl->slot = next;
            if (found > cap()) {
                give_up();
                T.ctl->slot = np2;
            }
            T.ctl->bail[0] = T.ctl->bail[1] = 0;
            T.ctl->cnt[0] = (uint32_t)b;
            T.ctl->cnt[1] = 0;
            T.ctl->cnt[2] = 0;
        }
        T.sync();
        const int32_t slot = (int32_t)T.get(&T.ctl->slot);
        if (slot >= np2) {  // the same for every thread of the team
            T.sync();       // no CTA leaves while another reads its shared memory
            break;
        }
        for (int i = threadIdx.x; i < g.bm_words / 4; i += blockDim.x)
            reinterpret_cast<uint4 *>(T.bm)[i] = make_uint4(0, 0, 0, 0);
        T.sync();
        const int32_t qi = g.qlist[slot];
        const uint32_t rk = a.rkey[qi];
        uint4 q[CPL];
        load_query<CPL>(a, a.queries + (size_t)qi * a.row_stride, q);

        // the lanes with `in` append their key to the items and to frontier list f (counter fc)
        auto append = [&](bool in, uint64_t k, uint32_t *f, uint32_t *fc) {
            const unsigned m = __ballot_sync(0xffffffffu, in);
            const int cnt = __popc(m);
            if (cnt == 0) return;
            const int p = __popc(m & lanemask_lt());
            const int room = kChunk - cfill;
            int64_t nb = 0;
            uint32_t f0 = 0;
            if (lane == 0) {
                if (cnt > room) nb = (int64_t)atomicAdd(g.tail, (unsigned long long)kChunk);
                if (fc) f0 = T.add(fc, (uint32_t)cnt);
            }
            nb = __shfl_sync(0xffffffffu, nb, 0);
            f0 = __shfl_sync(0xffffffffu, f0, 0);
            if (in) {
                const int64_t at = p < room ? cbase + cfill + p : nb + (p - room);
                if (at < g.cap) {
                    g.item_key[at] = k;
                    g.item_slot[at] = slot;
                }  // else the cursor says how long a list the host has to bring
                if (fc && f0 + p < g.fcap) f[f0 + p] = key_id(k);
            }
            if (cnt > room) {
                cbase = nb;
                cfill = cnt - room;
            } else {
                cfill += cnt;
            }
        };

        // F <- N: the query's full beam
        for (int i0 = (int)gw * 32; i0 < b; i0 += (int)stride * 32) {
            const int i = i0 + lane;
            const uint64_t k = i < b ? a.res_keys[(size_t)qi * b + i] : 0;
            if (i < b) {
                T.set(T.at(key_id(k)), 1u << (key_id(k) & 31));
                __stcg(fr + i, key_id(k));
            }
            append(i < b, k, nullptr, nullptr);
        }
        T.sync();
        uint32_t total = (uint32_t)b, L = 0;
        int32_t bail = 0;
        for (;; L++) {
            const uint32_t F = L == 0 ? (uint32_t)b : T.get(&T.ctl->cnt[L % 3]);
            if (L > 0) {
                total += F;
                bail = (int32_t)T.get(&T.ctl->bail[L & 1]);
                if (F > g.fcap && !bail) bail = kHandOver;
                if (F == 0 || bail) break;
            }
            const uint32_t *fin = fr + (size_t)(L & 1) * g.fcap;
            uint32_t *fout = fr + (size_t)((L & 1) ^ 1) * g.fcap;
            uint32_t *cout = &T.ctl->cnt[(L + 1) % 3];
            if (chief) {
                T.ctl->cnt[(L + 2) % 3] = 0;
                if (total >= g.bail_total && F >= g.bail_front && np2 - *(volatile int32_t *)g.done <= g.bail_slots)
                    T.ctl->bail[(L + 1) & 1] = kHandOver;
                if (F >= g.bail_front && *(volatile unsigned long long *)g.tail > cap() + g.slack) {
                    T.ctl->bail[(L + 1) & 1] = kStop;
                    give_up();
                }
            }
            // a small frontier: 2^sp warps share an item, each taking every 2^sp-th entry of its row, so that the
            // evaluations (several gather round trips a warp) spread over the team
            uint32_t sp = 0;
            while (sp < 3 && (F << (sp + 1)) <= stride && (stride >> sp) % 2 == 0) sp++;
            const uint32_t V = F << sp;
            const bool mine = ((lane ^ gw) & ((1u << sp) - 1)) == 0;  // strides are multiples of 2^sp
            // the warp's (shared) items gw, gw + stride, ...: ids are loaded two steps ahead, rows one ahead
            uint32_t row[4], idn[IW];
            auto load_ids = [&](uint32_t i) {
#pragma unroll
                for (int t = 0; t < IW; t++)
                    idn[t] = i + t * stride < V ? __ldcg(fin + ((i + t * stride) >> sp)) : kSent;
            };
            auto load_rows = [&]() {
#pragma unroll
                for (int t = 0; t < IW; t++)
#pragma unroll
                    for (int k = 0; k < RR; k++)
                        row[t * RR + k] = mine && idn[t] < (uint32_t)a.n && 32 * k + lane < R
                                              ? __ldg(a.adj + (size_t)idn[t] * R + 32 * k + lane) : kSent;
            };
            load_ids(gw);
            load_rows();
            load_ids(gw + IW * stride);
            int nc = 0;
            auto evaluate = [&](int n) {  // the last n <= 32 first-seen ids
                nc -= n;
                eval_candidates<DT, CPL, UN>(a, q, cid + nc, n, ckey);
                __syncwarp();
                const uint64_t k = lane < n ? ckey[lane] : kEmpty;
                append(lane < n && key_dk(k) <= rk, k, fout, cout);
                __syncwarp();
            };
            for (uint32_t i = gw; i < V; i += IW * stride) {
                uint32_t j[4], w[4], ad[4];
#pragma unroll
                for (int e = 0; e < 4; e++) {
                    j[e] = row[e];
                    w[e] = ~0u;
                    ad[e] = 0;
                    if (j[e] < (uint32_t)a.n) {
                        ad[e] = T.at(j[e]);
                        w[e] = T.word(ad[e]);
                    }
                }
                load_rows();
                load_ids(i + 2 * IW * stride);
#pragma unroll
                for (int e = 0; e < 4; e++) {
                    const uint32_t bit = 1u << (j[e] & 31);
                    bool fresh = !(w[e] & bit);
                    if (fresh) fresh = !(T.set(ad[e], bit) & bit);
                    const unsigned m = __ballot_sync(0xffffffffu, fresh);
                    if (fresh) cid[nc + __popc(m & lanemask_lt())] = j[e];
                    nc += __popc(m);
                }
                __syncwarp();
                while (nc >= 32) evaluate(32);
            }
            if (nc > 0) evaluate(nc);
            T.sync();
        }
        if (bail == kHandOver) {
            // hand over: the bitmap, and the next frontier (its points are results already).  One that has outgrown
            // its list is marked instead; the host takes all the query's results for it.
            const uint32_t F = T.get(&T.ctl->cnt[L % 3]);
            const uint32_t f = F > g.fcap ? 0u : F;
            if (chief) {
                const unsigned long long w = atomicAdd(g.hand_pend, (1ull << 32) + f);
                const uint32_t h = (uint32_t)(w >> 32), p = (uint32_t)w;
                const bool fits = h < (uint32_t)g.hand_cap && p + f <= g.pend_cap && p + f >= p;
                if (!fits) give_up();
                T.ctl->hand = fits ? (int32_t)h : -1;
                T.ctl->pend = p;
                if (fits) g.hand_of[slot] = (int32_t)h;
                if (fits && F > g.fcap) g.outgrown[h] = slot + 1;
            }
            T.sync();
            const int32_t h = (int32_t)T.get(&T.ctl->hand);
            if (h >= 0) {
                const uint32_t p = T.get(&T.ctl->pend);
                const uint32_t *fin = fr + (size_t)(L & 1) * g.fcap;
                for (uint32_t i = T.rank * blockDim.x + threadIdx.x; i < f; i += blockDim.x << T.log2) {
                    g.pend_key[p + i] = make_key(0, __ldcg(fin + i));
                    g.pend_slot[p + i] = slot;
                }
                uint32_t *out = g.hand_bits + (size_t)h * g.hand_words;
                for (int i = threadIdx.x; i < g.bm_words; i += blockDim.x) {
                    const int64_t w = ((int64_t)i << T.log2) + T.rank;
                    if (w < g.hand_words) out[w] = T.bm[i];
                }
            }
        }
        if (chief) {
            g.slot_count[slot] = (int32_t)total;
            a.res_count[qi] = (int32_t)total;
            atomicAdd(g.results, (unsigned long long)total);
            atomicAdd(g.done, 1);
            atomicMax(g.levels, (int32_t)L);
        }
        T.sync();  // everyone has read the control words: the next query may reset them
    }
    // the rest of the warp's chunk holds no items
    for (int t = cfill + lane; t < kChunk; t += 32)
        if (cbase + t < g.cap) g.item_slot[cbase + t] = -1;
}

template <int DT, int CPL, int RR>
rr_status bfs_r(const BfsArgs &g, const BfsShape &s, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(s.clusters << g.cl_log2));
    cfg.blockDim = dim3((unsigned)s.threads);
    cfg.dynamicSmemBytes = s.smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 1u << g.cl_log2;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    if (g.cl_log2 > 0) {
        cfg.attrs = at;
        cfg.numAttrs = 1;
    }
    auto k = g.cl_log2 == 0 ? bfs_kernel<DT, CPL, RR, false> : bfs_kernel<DT, CPL, RR, true>;
    if (rr_status e = allow_smem((const void *)k, s.smem)) return e;
    RR_CUDA(cudaLaunchKernelEx(&cfg, k, g));
    note_launch();
    return RR_OK;
}

template <int DT, int CPL>
rr_status bfs_t(const BfsArgs &g, const BfsShape &s, cudaStream_t st) {
    if (g.s.R <= 32) return bfs_r<DT, CPL, 1>(g, s, st);
    if (g.s.R <= 64) return bfs_r<DT, CPL, 2>(g, s, st);
    return bfs_r<DT, CPL, 4>(g, s, st);
}

}  // namespace

}  // namespace rr
