// k_beam_cta.cu -- the beam phase (see k_beam.cu) by a CTA per query, for batches too small to fill the chip with a
// warp per query.
//
// There the time is the chain of one query's visits, each a row, the gather of its unseen neighbours' vectors and the
// merge behind one another.  The chain is shortened by looking ahead: the K closest unvisited points of B are known,
// so their rows' unseen neighbours are evaluated together, a warp (or, with K below the warps, several) per parent.
// Parent k is then visited in this step exactly if no neighbour found under the parents before it is as close to q as
// it is: B up to it, and with it every choice of Alg. 1 and the early stop on d_visited or d_top1, is that of one
// visit at a time (later keys enter behind it, and a point stays in B while fewer than b are closer).  Neighbours
// of the others were evaluated for nothing and are forgotten.  K doubles while all of it holds and falls to one more
// than what held.  The rows of the next points in line are loaded into shared memory during the evaluation.
//
// The seen table is the two-way lossy one of k_beam.cu, shared by the warps: it is read in one phase of a step and
// written in another, and racing writers can only lose an id, which costs a repeated evaluation.
//
// Measured (GB300, beam phase, a warp per query -> this): 1 query, beam 192, 10^6 x 128 u8, R = 64: 175 -> 110 us.
// By warps a query, on five indexes (u8 128 B, R = 64 and 128; i8 256 B, R = 24; fp32 800 B, R = 64, and 2 KB, R = 128),
// beams 32 to 512, with and without early stop, the warp form's time over this one's:
//   8 (up to 304 queries)    1.2 to 2.7 times up to beam 256, 1.0 to 2.1 beyond (1.0: 8-bit, one query)
//   4 (305 to 608)           1.1 to 1.9; one of the cases loses: i8, early stop, beam 512, 0.94
//   2 (609 to 1,216)         8-bit 1.02 to 1.21 up to beam 128, 0.92 to 1.04 at 160 to 256, 0.80 to 0.94 beyond;
//                            fp32 1.08 to 1.46 up to beam 256, 0.92 to 1.09 beyond
// At 2,048 queries a warp each fills the chip (2*10^5 x 128 u8, R = 32, beam 64 / 192): 651 / 1,317 us against
// 659 / 1,593.  Bound: the chain of steps (row, gather, six barriers).
#include <algorithm>

#include "rr_common.cuh"

namespace rr {

namespace {

constexpr int kMaxW = 8;  // warps of a CTA = parents of a step

constexpr int kHashLg = 11;  // unless the caller sets seen_log2

__host__ __device__ inline int even(int x) { return (x + 1) & ~1; }
__host__ __device__ inline size_t cta_smem_bytes(int b, int R, int W, int hlg) {
    return (size_t)2 * b * 8 + (size_t)W * R * 8 * 2 + (size_t)even(W * R) * 4 * 3 + ((size_t)4 << hlg);
}

__device__ __forceinline__ int lower_bound_or1(const uint64_t *a, int n, uint64_t k1) {
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if ((a[mid] | 1ull) < k1) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

template <int DT, int CPL>
__global__ void __launch_bounds__(32 * kMaxW, 2) beam_cta_kernel(SearchArgs a, int hlg) {
    extern __shared__ __align__(16) uint8_t smem_raw[];
    constexpr int UN = CPL == 1 ? 8 : (CPL == 2 ? 4 : 2);
    __shared__ uint64_t pkey[2 * kMaxW];          // the parents, then the next points in line
    __shared__ int ppos[2 * kMaxW];
    __shared__ uint32_t mind[kMaxW], rowid[kMaxW];
    __shared__ int s_K, s_got, s_ns[2], s_nu[2], s_stop;
    const int lane = lane_id(), warp = threadIdx.x >> 5, tid = threadIdx.x, T = blockDim.x, W = T >> 5;
    const int64_t qi = blockIdx.x;
    const int R = a.R, b = a.beam, H = 1 << hlg;
    uint64_t *B = reinterpret_cast<uint64_t *>(smem_raw), *B2 = B + b;
    uint64_t *ckeys = B2 + b, *skey = ckeys + W * R;  // candidates (later: sorted survivors), survivors
    uint32_t *cids = reinterpret_cast<uint32_t *>(skey + W * R);
    int32_t *slb = reinterpret_cast<int32_t *>(cids + even(W * R));
    uint32_t *rows = reinterpret_cast<uint32_t *>(slb + even(W * R));
    uint32_t *hash = rows + even(W * R);
    uint64_t *ckey = ckeys + warp * R;
    uint32_t *cid = cids + warp * R;
    int32_t *lbs = reinterpret_cast<int32_t *>(cids);  // insertion points of the sorted survivors

    uint4 q[CPL];
    load_query<CPL>(a, a.queries + (size_t)qi * a.row_stride, q);
    const uint32_t rk = a.rkey[qi], ek = a.eskey[qi];
    for (int i = tid; i < H; i += T) hash[i] = kSent;
    if (tid < W) rowid[tid] = kSent;
    const uint32_t dk0 = eval_one<DT, CPL>(a, q, a.start);
    __syncthreads();
    if (tid == 0) {
        B[0] = make_key(dk0, a.start);
        hash[hslot(a.start, hlg - 1) << 1] = a.start;
        s_stop = 0;
    }
    __syncthreads();
    int nb = 1, nvis = 0, Kt = 1;
    int cur = 0;  // every entry before it is visited
    for (int it = 0;; it ^= 1) {
        if (warp == 0) {
            // the next unvisited points: up to Kt parents, and those in line after them
            int got = 0;
            for (int t0 = cur; t0 < nb && got < Kt + W; t0 += 32) {
                const int t = t0 + lane;
                const uint64_t k = t < nb ? B[t] : 1ull;
                const unsigned m = __ballot_sync(0xffffffffu, !(k & 1ull));
                if (got == 0) cur = m ? t0 + __ffs(m) - 1 : min(t0 + 32, nb);
                const int r = got + __popc(m & lanemask_lt());
                if (!(k & 1ull) && r < Kt + W) {
                    pkey[r] = k;
                    ppos[r] = t;
                }
                got = min(Kt + W, got + __popc(m));
            }
            __syncwarp();
            int K = min(got, Kt);
            if (a.use_es && K > 0) {
                const uint32_t d0 = key_dk(B[0]);
                const bool fire = lane < K && d0 > rk && nvis + lane >= a.es_vl &&
                                  (a.es_metric == RR_ES_TOP1 ? d0 : key_dk(pkey[lane & (kMaxW - 1)])) > ek;
                const unsigned m = __ballot_sync(0xffffffffu, fire);
                if (m) K = __ffs(m) - 1;
                if (K == 0 && lane == 0) s_stop = 1;
            }
            if (K > 0 && nvis + K > a.iter_limit) {  // cannot happen for a validated index
                K = (int)(a.iter_limit - nvis);
                if (K <= 0 && lane == 0) atomicExch(a.error, 1);
                K = max(K, 0);
            }
            if (lane == 0) {
                s_K = K;
                s_got = got;
                s_ns[it] = s_nu[it] = 0;
            }
        }
        __syncthreads();
        const int K = s_K;
        if (K == 0) break;
        // 2^lg groups of G warps, a group per parent, a warp per part of its row
        const int lg = K <= 1 ? 0 : 32 - __clz(K - 1);
        const int G = W >> lg, par = warp / G;
        uint32_t pre[4], pre_id = kSent;
        if (K + warp < s_got) pre_id = key_id(pkey[K + warp]);
        int nc = 0;
        if (par < K) {
            const uint32_t p = key_id(pkey[par]);
            const int part = (R + G - 1) / G, e0 = (warp % G) * part, e1 = min(R, e0 + part);
            const unsigned hit = __ballot_sync(0xffffffffu, lane < W && rowid[lane & (kMaxW - 1)] == p);
            const uint32_t *row = hit ? rows + (__ffs(hit) - 1) * R : a.adj + (size_t)p * R;
            uint32_t j4[4];
#pragma unroll
            for (int k = 0; k < 4; k++) j4[k] = e0 + 32 * k + lane < e1 ? row[e0 + 32 * k + lane] : kSent;
#pragma unroll
            for (int k = 0; k < 4; k++)
                pre[k] = pre_id != kSent && 32 * k + lane < R ? __ldg(a.adj + (size_t)pre_id * R + 32 * k + lane) : kSent;
#pragma unroll
            for (int k = 0; k < 4; k++) {
                if (e0 + 32 * k >= e1) break;
                const uint32_t j = j4[k];
                bool v = j < (uint32_t)a.n;  // also drops the padding
                if (v) {
                    const uint32_t sl = hslot(j, hlg - 1) << 1;
                    v = hash[sl] != j && hash[sl + 1] != j;
                }
                const unsigned m = __ballot_sync(0xffffffffu, v);
                if (v) cid[nc + __popc(m & lanemask_lt())] = j;
                nc += __popc(m);
            }
            __syncwarp();
            uint32_t mn = 0xffffffffu;
            if (nc > 0) {
                eval_candidates<DT, CPL, UN>(a, q, cid, nc, ckey);
                __syncwarp();
                for (int c = lane; c < nc; c += 32) mn = min(mn, key_dk(ckey[c]));
                mn = __reduce_min_sync(0xffffffffu, mn);
            }
            if (lane == 0) mind[warp] = mn;
        } else {
#pragma unroll
            for (int k = 0; k < 4; k++)
                pre[k] = pre_id != kSent && 32 * k + lane < R ? __ldg(a.adj + (size_t)pre_id * R + 32 * k + lane) : kSent;
        }
        __syncthreads();
        int nk = 1;
        for (uint32_t mn = 0xffffffffu; nk < K; nk++) {
            for (int w = (nk - 1) * G; w < nk * G; w++) mn = min(mn, mind[w]);
            if (mn <= key_dk(pkey[nk])) break;
        }
        // V <- V u the first nk parents; their neighbours are seen
        const uint64_t last = nb == b ? (B[b - 1] | 1ull) : kEmpty;
        if (par < nk) {
            for (int c0 = 0; c0 < nc; c0 += 32) {
                const int c = c0 + lane;
                const uint64_t k = c < nc ? ckey[c] : kEmpty;
                if (c < nc) {
                    const uint32_t sl = hslot(key_id(k), hlg - 1) << 1;
                    hash[sl + 1] = hash[sl];
                    hash[sl] = key_id(k);
                }
                const bool keep = c < nc && (k | 1ull) < last;
                const unsigned m = __ballot_sync(0xffffffffu, keep);
                if (m) {
                    int at = 0;
                    if (lane == 0) at = atomicAdd(&s_ns[it], __popc(m));
                    at = __shfl_sync(0xffffffffu, at, 0);
                    if (keep) skey[at + __popc(m & lanemask_lt())] = k;
                }
            }
        }
#pragma unroll
        for (int k = 0; k < 4; k++)
            if (32 * k + lane < R) rows[warp * R + 32 * k + lane] = pre[k];
        if (lane == 0) rowid[warp] = pre_id;
        __syncthreads();
        if (warp == 0 && lane < nk) B[ppos[lane]] |= 1ull;  // after every read of B's last key
        nvis += nk;
        Kt = nk == K ? min(W, 2 * nk) : nk + 1;
        const int ns = s_ns[it];
        __syncwarp();
        if (ns == 0) continue;
        // not in B already (the table forgets) and the first of its kind (two parents of a step share neighbours)
        for (int c = tid; c < ns; c += T) {
            const uint64_t k = skey[c];
            const int lb = lower_bound_or1(B, nb, k | 1ull);
            bool ok = !(lb < nb && (B[lb] | 1ull) == (k | 1ull));
            for (int t = 0; t < c && ok; t++) ok = skey[t] != k;
            slb[c] = ok ? lb : -1;
        }
        __syncthreads();
        for (int c = tid; c < ns; c += T) {
            const int lb = slb[c];
            if (lb < 0) continue;
            const uint64_t k = skey[c];
            int r = 0;
            for (int t = 0; t < ns; t++) r += slb[t] >= 0 && skey[t] < k;
            ckeys[r] = k;
            lbs[r] = lb;
            atomicAdd(&s_nu[it], 1);
        }
        __syncthreads();
        const int nu = s_nu[it];
        if (nu == 0) continue;
        // B <- top-b(B u survivors)
        for (int t = tid; t < nb; t += T) {
            const uint64_t k = B[t];
            const int pos = t + lower_bound_or1(ckeys, nu, k | 1ull);
            if (pos < b) B2[pos] = k;
        }
        for (int t = tid; t < nu; t += T)
            if (lbs[t] + t < b) B2[lbs[t] + t] = ckeys[t];
        if (warp == 0) cur = min(cur, lbs[0]);
        __syncthreads();
        nb = min(b, nb + nu);
        uint64_t *t = B;
        B = B2;
        B2 = t;
    }
    // N = {n in B : d(n, q) <= r}, a prefix
    int cnt = 0;
    for (int hi = nb; cnt < hi;) {
        const int mid = (cnt + hi) >> 1;
        if (key_dk(B[mid]) <= rk) cnt = mid + 1;
        else hi = mid;
    }
    uint64_t *out = a.res_keys + (size_t)qi * b;
    for (int i = tid; i < cnt; i += T) out[i] = B[i] & ~1ull;
    if (tid == 0) {
        a.res_count[qi] = cnt;
        uint8_t f = s_stop ? RR_FLAG_EARLY_STOPPED : 0;
        if (a.phase2 && cnt == b) {
            f |= RR_FLAG_PHASE2;
            a.p2_list[atomicAdd(a.p2_count, 1)] = (int32_t)qi;
        }
        a.flags[qi] = f;
    }
}

template <int DT, int CPL>
rr_status launch_t(const SearchArgs &a, cudaStream_t st) {
    auto k = beam_cta_kernel<DT, CPL>;
    const int W = a.nq <= kBeamCta8 ? 8 : (a.nq <= kBeamCta4 ? 4 : 2);
    const int hlg = a.hash_lg > 0 ? a.hash_lg : kHashLg;
    const size_t smem = cta_smem_bytes(a.beam, a.R, W, hlg);
    if (rr_status e = allow_smem((const void *)k, smem)) return e;
    k<<<(unsigned)a.nq, 32 * W, smem, st>>>(a, hlg);
    RR_CUDA(cudaGetLastError());
    note_launch();
    return RR_OK;
}

}  // namespace

// The CTA form: exact traversal, one parent per visit, no exact counters (its evaluation counts would differ), an
// early stop that the lookahead can foresee, and beams long enough to have points in line (beam 16: 172 -> 186 us,
// beam 64: 521 -> 400 us at 64 queries).  With two warps a query only beams that these merge as fast as one warp does
// (table above).
bool beam_cta(const SearchArgs &a, int dtype_code) {
    return a.nq <= (a.beam <= (dtype_code == DT_F32 ? kBeamCta2F32 : kBeamCta2Int) ? kBeamCta2 : kBeamCta4) &&
           a.beam >= kBeamCtaBeam && a.expand <= 1 && !a.count_bits && !a.stats && a.prec == RR_PREC_EXACT &&
           (!a.use_es || a.es_metric == RR_ES_VISITED || a.es_metric == RR_ES_TOP1);
}

rr_status launch_beam_cta(const SearchArgs &a, cudaStream_t st, int dtype_code) {
    const int cpl = (a.row_chunks + 31) / 32;
    switch (dtype_code) {
        case DT_U8: return launch_t<DT_U8, 1>(a, st);
        case DT_I8: return launch_t<DT_I8, 1>(a, st);
        case DT_F32:
            if (cpl <= 1) return launch_t<DT_F32, 1>(a, st);
            if (cpl <= 2) return launch_t<DT_F32, 2>(a, st);
            return launch_t<DT_F32, 4>(a, st);
    }
    set_error("beam phase: unsupported element type %d", dtype_code);
    return RR_EINVAL;
}

}  // namespace rr
