// k_doubling.cu -- Alg. 3 DoublingSearch for the queries whose first beam
// search returned a full beam of in-range points (|N| = b, lambda = 1).
//
// Rounds are host-driven: round k runs Alg. 1 with beam b_k = b_0 * 2^(k-1)
// from B = S_k (trimming S_k to its b_k closest up front is equivalent: the
// first visit is the closest point of S_k either way, and top-b(S u X) =
// top-b(top-b(S) u X) at the first trim), with a fresh V.  Round 1 is
// re-run here from S = {start}, so the round kernel owns the whole per-query
// state.  Then S <- S u V (the b_max smallest keys are all any later round
// can use) and b <- 2b while |N| = b.
//
// Per query and round, one warp.  The beam can be tens of thousands of keys,
// so it lives in global memory (L2-resident) as a sorted array M, with a small
// sorted insertion buffer I in shared memory; the logical beam is the b
// smallest keys of M u I, tracked through their b-th key tau.  New keys enter
// I only if they are below tau; I is merged into M when full.  An exact
// per-round bitmap of evaluated ids replaces the visited filter (an id that is
// seen again is either in the beam or was trimmed, and a trimmed id can never
// re-enter: see the beam kernel), so no id is evaluated twice in a round.
#include "rr_common.cuh"

namespace rr {

namespace {

constexpr int KI = 256;  // insertion buffer entries

__device__ __forceinline__ int lb_or1(const uint64_t *a, int n, uint64_t k1) {
    int lo = 0, hi = n;
    while (lo < hi) {
        int mid = (lo + hi) >> 1;
        if ((a[mid] | 1ull) < k1) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// number of a[t] with (a[t] | 1) <= k1
__device__ __forceinline__ int ub_or1(const uint64_t *a, int n, uint64_t k1) {
    int lo = 0, hi = n;
    while (lo < hi) {
        int mid = (lo + hi) >> 1;
        if ((a[mid] | 1ull) <= k1) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// (key | 1) of the element of rank b-1 (0-based) of the sorted union M u I,
// or kEmpty when the union has fewer than b keys.  Serial (one lane).
__device__ uint64_t kth_or1(const uint64_t *M, int nM, const uint64_t *I, int nI, int b) {
    if (nM + nI < b) return kEmpty;
    int lo = max(0, b - nI), hi = min(b, nM);
    // largest i in [lo, hi] with: i == 0 || b - i >= nI || M[i-1] < I[b-i]
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        bool ok = (b - mid >= nI) || ((M[mid - 1] | 1ull) < (I[b - mid] | 1ull));
        if (ok) lo = mid;
        else hi = mid - 1;
    }
    int i = lo, j = b - lo;
    uint64_t x = i > 0 ? (M[i - 1] | 1ull) : 0ull;
    uint64_t y = j > 0 ? (I[j - 1] | 1ull) : 0ull;
    return x > y ? x : y;
}

struct RSmem {
    uint64_t *I, *I2, *ckey, *skey;
    uint32_t *cid;
};

// per warp, rounded to 16 bytes so that every warp's 8-byte arrays stay aligned for any degree R
__host__ __device__ inline size_t round_smem_bytes(int R) {
    return ((size_t)2 * KI * 8 + (size_t)2 * R * 8 + (size_t)R * 4 + 15) & ~(size_t)15;
}

template <int DT, int CPL>
__global__ void __launch_bounds__(128) round_kernel(DoublingRound d) {
    extern __shared__ __align__(16) uint8_t smem_raw[];
    constexpr int UN = CPL == 1 ? 8 : (CPL == 2 ? 4 : 2);
    const SearchArgs &a = d.s;
    const int lane = lane_id();
    const int warp = threadIdx.x >> 5;
    const int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp;
    if (i >= d.na) return;
    const int R = a.R;
    const int b = a.beam;
    uint8_t *base = smem_raw + (size_t)warp * round_smem_bytes(R);
    RSmem s;
    s.I = reinterpret_cast<uint64_t *>(base);
    s.I2 = s.I + KI;
    s.ckey = s.I2 + KI;
    s.skey = s.ckey + R;
    s.cid = reinterpret_cast<uint32_t *>(s.skey + R);

    const int32_t slot = d.act[i];
    const int32_t qi = d.qlist[slot];
    constexpr bool LP = is_lowp(DT);
    uint4 q[CPL];
    float qf[16];
    float qn2 = 0.f;
    if constexpr (LP) {
        load_query_lp<DT>(a, reinterpret_cast<const float *>(a.queries + (size_t)qi * a.row_stride), qf);
        qn2 = query_norm2_lp(a, qf);
    } else {
        load_query<CPL>(a, a.queries + (size_t)qi * a.row_stride, q);
    }
    const uint32_t rk = a.rkey[qi], ek = a.eskey[qi];
    const uint32_t rks = LP ? slack_key(a, rk, qn2) : rk;  // approximate keys above rks are out of range
    uint64_t *M = d.bA + (size_t)i * b;
    uint64_t *M2 = d.bB + (size_t)i * b;
    uint64_t *V = d.v + (size_t)i * d.v_cap;
    // warm restart: the bitmap of every id this query ever evaluated lives on across rounds (per slot)
    uint32_t *seen = d.seen + (size_t)(d.warm ? slot : i) * d.seen_words;
    uint64_t *EV = d.warm ? d.ev + (size_t)i * d.ev_cap : nullptr;
    int nev = 0;
    uint32_t *cbits = a.count_bits ? a.count_bits + (size_t)qi * a.words_per_q : nullptr;
    int evals = 0, distinct = 0;

    // B <- top-b(S)
    int nM;
    if (d.first) {
        uint32_t dk0;
        if constexpr (LP) dk0 = eval_one_lp<DT>(a, qf, qn2, a.start);
        else dk0 = eval_one<DT, CPL>(a, q, a.start);
        if (lane == 0) {
            M[0] = make_key(dk0, a.start);
            mark_bit(seen, a.start);
            if (EV) EV[0] = make_key(dk0, a.start);
        }
        nev = EV ? 1 : 0;
        nM = 1;
        evals = 1;
    } else if (d.warm) {
        // B <- the b closest points of E, visited ones still marked (they are not visited again); every id
        // of E is in seen already: one outside these b can never enter the beam of this round
        nM = min(b, d.s_cnt[i]);
        const uint64_t *S = d.s_old + (size_t)i * d.s_cap;
        for (int t = lane; t < nM; t += 32) M[t] = S[t];
    } else {
        nM = min(b, d.s_cnt[i]);
        const uint64_t *S = d.s_old + (size_t)i * d.s_cap;
        for (int t = lane; t < nM; t += 32) {
            uint64_t k = S[t] & ~1ull;
            M[t] = k;
            mark_bit(seen, key_id(k));
        }
    }
    __syncwarp();
    int nI = 0, cM = 0, nvis = 0;
    bool stopped = false, overflow = false;
    uint64_t tau = (nM >= b) ? (M[b - 1] | 1ull) : kEmpty;
    int64_t guard = 0;

    for (;;) {
        // first unvisited key of M from the cursor
        for (;;) {
            int t = cM + lane;
            bool un = t < nM && !(M[t] & 1ull);
            unsigned m = __ballot_sync(0xffffffffu, un);
            if (m) { cM += __ffs(m) - 1; break; }
            cM += 32;
            if (cM >= nM) { cM = nM; break; }
        }
        uint64_t kM = cM < nM ? M[cM] : kEmpty;
        int jI = -1;
        for (int b0 = 0; b0 < nI; b0 += 32) {
            int t = b0 + lane;
            bool un = t < nI && !(s.I[t] & 1ull);
            unsigned m = __ballot_sync(0xffffffffu, un);
            if (m) { jI = b0 + __ffs(m) - 1; break; }
        }
        uint64_t kI = jI >= 0 ? s.I[jI] : kEmpty;
        const bool fromI = (kI | 1ull) < (kM | 1ull);
        const uint64_t pk = fromI ? kI : kM;
        if (pk == kEmpty || (pk | 1ull) > tau) break;  // B \ V is empty
        if (a.use_es) {
            uint64_t mn = M[0] | 1ull;
            if (nI > 0 && (s.I[0] | 1ull) < mn) mn = s.I[0] | 1ull;
            if (key_dk(mn) > rks && nvis >= a.es_vl && key_dk(pk) > ek) { stopped = true; break; }
        }
        if (++guard > a.iter_limit) {
            if (lane == 0) atomicExch(a.error, 2);
            break;
        }
        if (nvis >= d.v_cap) { overflow = true; break; }
        __syncwarp();
        if (lane == 0) {
            if (fromI) s.I[jI] = pk | 1ull;
            else M[cM] = pk | 1ull;
            V[nvis] = pk & ~1ull;
        }
        nvis++;
        const uint32_t p = key_id(pk);
        const uint32_t *row = a.adj + (size_t)p * R;
        int nc = 0;
        for (int e0 = 0; e0 < R; e0 += 32) {
            int e = e0 + lane;
            uint32_t j = e < R ? __ldg(row + e) : kSent;
            bool v = j < (uint32_t)a.n && mark_bit(seen, j);
            unsigned m = __ballot_sync(0xffffffffu, v);
            if (v) s.cid[nc + __popc(m & lanemask_lt())] = j;
            nc += __popc(m);
        }
        __syncwarp();
        if (nc == 0) continue;
        evals += nc;
        if constexpr (LP) eval_candidates_lp<DT, DT == DT_FP8 ? 4 : 8>(a, qf, qn2, s.cid, nc, s.ckey);
        else eval_candidates<DT, CPL, UN>(a, q, s.cid, nc, s.ckey);
        __syncwarp();
        if (EV) {
            // E <- E u the new evaluations (kept for the rounds after this one)
            if (nev + nc > d.ev_cap) { overflow = true; break; }
            for (int c = lane; c < nc; c += 32) EV[nev + c] = s.ckey[c];
            nev += nc;
        }
        if (cbits) {
            int dd = 0;
            for (int c = lane; c < nc; c += 32) dd += mark_bit(cbits, s.cid[c]);
            distinct += dd;
        }
        // keys below tau enter the beam
        int ns = 0;
        for (int c0 = 0; c0 < nc; c0 += 32) {
            int c = c0 + lane;
            uint64_t k = c < nc ? s.ckey[c] : kEmpty;
            bool keep = c < nc && (k | 1ull) < tau;
            unsigned m = __ballot_sync(0xffffffffu, keep);
            if (keep) s.skey[ns + __popc(m & lanemask_lt())] = k;
            ns += __popc(m);
        }
        __syncwarp();
        if (ns == 0) continue;
        for (int c = lane; c < ns; c += 32) {
            uint64_t k = s.skey[c];
            int r = 0;
            for (int t = 0; t < ns; t++) r += s.skey[t] < k;
            s.ckey[r] = k;  // survivors sorted
        }
        __syncwarp();
        if (nI + ns > KI) {
            // flush: M2 <- top-b(M u I)
            for (int t = lane; t < nM; t += 32) {
                uint64_t k = M[t];
                int pos = t + lb_or1(s.I, nI, k | 1ull);
                if (pos < b) M2[pos] = k;
            }
            for (int t = lane; t < nI; t += 32) {
                uint64_t k = s.I[t];
                int pos = t + lb_or1(M, nM, k | 1ull);
                if (pos < b) M2[pos] = k;
            }
            int posM = cM < nM ? cM + lb_or1(s.I, nI, M[cM] | 1ull) : 0x7fffffff;
            int jU = -1;
            for (int b0 = 0; b0 < nI; b0 += 32) {
                int t = b0 + lane;
                bool un = t < nI && !(s.I[t] & 1ull);
                unsigned m = __ballot_sync(0xffffffffu, un);
                if (m) { jU = b0 + __ffs(m) - 1; break; }
            }
            int posI = jU >= 0 ? jU + lb_or1(M, nM, s.I[jU] | 1ull) : 0x7fffffff;
            __syncwarp();
            nM = min(b, nM + nI);
            nI = 0;
            cM = min(min(posM, posI), nM);
            uint64_t *t = M;
            M = M2;
            M2 = t;
        }
        // I <- I u survivors (sorted merge into I2, then copy back)
        for (int t = lane; t < nI; t += 32) {
            uint64_t k = s.I[t];
            s.I2[t + lb_or1(s.ckey, ns, k | 1ull)] = k;
        }
        for (int t = lane; t < ns; t += 32) {
            uint64_t k = s.ckey[t];
            s.I2[t + lb_or1(s.I, nI, k | 1ull)] = k;
        }
        __syncwarp();
        nI += ns;
        for (int t = lane; t < nI; t += 32) s.I[t] = s.I2[t];
        __syncwarp();
        // tau <- b-th smallest of M u I; drop I keys beyond it
        uint64_t nt = 0;
        if (lane == 0) nt = kth_or1(M, nM, s.I, nI, b);
        tau = __shfl_sync(0xffffffffu, nt, 0);
        if (tau != kEmpty) nI = ub_or1(s.I, nI, tau);
        __syncwarp();
    }
    // final B = top-b(M u I)
    if (nI > 0) {
        for (int t = lane; t < nM; t += 32) {
            uint64_t k = M[t];
            int pos = t + lb_or1(s.I, nI, k | 1ull);
            if (pos < b) M2[pos] = k;
        }
        for (int t = lane; t < nI; t += 32) {
            uint64_t k = s.I[t];
            int pos = t + lb_or1(M, nM, k | 1ull);
            if (pos < b) M2[pos] = k;
        }
        __syncwarp();
        nM = min(b, nM + nI);
        uint64_t *t = M;
        M = M2;
        M2 = t;
    }
    // N = {n in B : d <= r} (low precision: exact fp32 recheck of the prefix within r + slack)
    int cnt = 0;
    for (int b0 = 0; b0 < nM; b0 += 32) {
        int t = b0 + lane;
        bool in = t < nM && key_dk(M[t]) <= rks;
        cnt += __popc(__ballot_sync(0xffffffffu, in));
    }
    if constexpr (LP) {
        evals += cnt;
        cnt = exact_filter_sort<CPL, UN>(a, qi, M, cnt, rk, s.cid, s.ckey, R);
    }
    const bool cont = !stopped && !overflow && cnt == b && !d.last;
    if (!cont) {
        // finished: append N to the result items
        unsigned long long basepos = 0;
        if (lane == 0 && cnt > 0) basepos = atomicAdd(d.tail, (unsigned long long)cnt);
        basepos = __shfl_sync(0xffffffffu, basepos, 0);
        int written = 0;
        for (int t = lane; t < cnt; t += 32) {
            unsigned long long pos = basepos + t;
            if (pos < (unsigned long long)d.cap) {
                d.item_key[pos] = M[t] & ~1ull;
                d.item_slot[pos] = slot;
                written++;
            }
        }
        for (int o = 16; o > 0; o >>= 1) written += __shfl_xor_sync(0xffffffffu, written, o);
        if (lane == 0) {
            d.slot_count[slot] = written;
            d.slot_trunc[slot] = (written < cnt || overflow || (d.last && cnt == b && !stopped)) ? 1 : 0;
        }
    }
    if (cbits) {
        for (int o = 16; o > 0; o >>= 1) distinct += __shfl_xor_sync(0xffffffffu, distinct, o);
    }
    if (lane == 0) {
        d.status[i] = cont ? 1 : 0;
        d.nv[i] = nvis;
        if (d.nev) d.nev[i] = nev;
        if (a.stats) {
            rr_query_stats *st = a.stats + qi;
            if (d.first) {
                // round 1 repeats the beam phase exactly: replace its counters
                st->visits_beam = nvis;
                st->rounds = 1;
                st->evals = evals;  // distinct: the same ids as the beam phase, already counted
            } else {
                st->visits_beam += nvis;
                st->rounds += 1;
                st->evals += evals;
                st->distinct += distinct;
            }
            st->final_beam = b;
        }
    }
}

// The same round by a CTA per query, for rounds with few active queries: there the time is that of the longest
// query, a chain of b and more visits in order, each a row, its seen words, the vectors and the merge behind one
// another (2^15 visits in all for a query with 10^4 results).  Looking ahead shortens the chain: the next K
// unvisited keys of the beam are known, so their rows are read and their unseen neighbours evaluated together, a
// warp (or, with K below the warps, several) per parent.  Parent k is then visited in this step exactly if no
// neighbour found under the parents before it is as close as it is: the beam's order up to it, and so every choice
// of Alg. 1, is that of one visit at a time (later keys enter behind it, and a key stays in the beam while fewer
// than b are below it).  The rest were evaluated for nothing and stay unmarked.  K grows while all of it holds.
// Measured (GB300, 41 doubling queries of 10^6 x 128 u8, 10 rounds up to b = 8,192, 41 K results): 45.2 -> 16.2 ms.
// Bound: still the longest query's chain of steps, each about five dependent memory round trips and barriers.
constexpr int CW = 8;  // warps, and the most parents of a step

// (key | 1) of rank b-1 of M u I and the number of keys of I up to it, as kth_or1, with a warp (32 probes a step)
__device__ uint64_t warp_kth_or1(const uint64_t *M, int nM, const uint64_t *I, int nI, int b, int *jI) {
    *jI = nI;
    if (nM + nI < b) return kEmpty;
    int lo = max(0, b - nI), hi = min(b, nM);
    while (lo < hi) {
        const int step = (hi - lo + 31) >> 5;
        const int mid = lo + (lane_id() + 1) * step;
        const bool ok = mid <= hi && ((b - mid >= nI) || ((M[mid - 1] | 1ull) < (I[b - mid] | 1ull)));
        const int c = __popc(__ballot_sync(0xffffffffu, ok));  // ok falls once
        lo += c * step;
        hi = min(hi, lo + step - 1);
    }
    const int i = lo, j = b - lo;
    const uint64_t x = i > 0 ? (M[i - 1] | 1ull) : 0ull;
    const uint64_t y = j > 0 ? (I[j - 1] | 1ull) : 0ull;
    *jI = j;
    return x > y ? x : y;
}

__host__ __device__ inline int cta_buffer_keys(int R) { return CW * R < 256 ? 256 : CW * R; }
__host__ __device__ inline size_t round_cta_smem_bytes(int R) {
    return (size_t)2 * cta_buffer_keys(R) * 8 + (size_t)CW * R * (8 + 8 + 4);
}

template <int DT, int CPL>
__global__ void __launch_bounds__(32 * CW) round_cta_kernel(DoublingRound d) {
    extern __shared__ __align__(16) uint8_t smem_raw[];
    constexpr int UN = CPL == 1 ? 8 : (CPL == 2 ? 4 : 2);
    __shared__ uint64_t pkey[CW], selk[2 * CW], s_tau;
    __shared__ int ppos[CW], selp[2 * CW];
    __shared__ uint32_t mind[CW];
    __shared__ int s_K, s_nI, s_ns[2], s_end, s_cnt;
    __shared__ unsigned long long s_base;
    __shared__ int s_nev;
    const SearchArgs &a = d.s;
    const int lane = lane_id(), warp = threadIdx.x >> 5, tid = threadIdx.x, T = 32 * CW;
    const int64_t i = blockIdx.x;
    const int R = a.R, b = a.beam, ki = cta_buffer_keys(R);
    uint64_t *I = reinterpret_cast<uint64_t *>(smem_raw), *I2 = I + ki;
    uint64_t *ckeys = I2 + ki, *skey = ckeys + CW * R;
    uint64_t *ckey = ckeys + warp * R;
    uint32_t *cid = reinterpret_cast<uint32_t *>(skey + CW * R) + warp * R;

    const int32_t slot = d.act[i];
    const int32_t qi = d.qlist[slot];
    constexpr bool LP = is_lowp(DT);
    uint4 q[CPL];
    float qf[16];
    float qn2 = 0.f;
    if constexpr (LP) {
        load_query_lp<DT>(a, reinterpret_cast<const float *>(a.queries + (size_t)qi * a.row_stride), qf);
        qn2 = query_norm2_lp(a, qf);
    } else {
        load_query<CPL>(a, a.queries + (size_t)qi * a.row_stride, q);
    }
    const uint32_t rk = a.rkey[qi], ek = a.eskey[qi];
    const uint32_t rks = LP ? slack_key(a, rk, qn2) : rk;  // approximate keys above rks are out of range
    uint64_t *M = d.bA + (size_t)i * b;
    uint64_t *M2 = d.bB + (size_t)i * b;
    uint64_t *V = d.v + (size_t)i * d.v_cap;
    uint32_t *seen = d.seen + (size_t)(d.warm ? slot : i) * d.seen_words;
    uint64_t *EV = d.warm ? d.ev + (size_t)i * d.ev_cap : nullptr;

    // B <- top-b(S), as in round_kernel
    int nM;
    if (d.first) {
        uint32_t dk0;
        if constexpr (LP) dk0 = eval_one_lp<DT>(a, qf, qn2, a.start);
        else dk0 = eval_one<DT, CPL>(a, q, a.start);
        if (tid == 0) {
            M[0] = make_key(dk0, a.start);
            mark_bit(seen, a.start);
            if (EV) EV[0] = make_key(dk0, a.start);
        }
        nM = 1;
    } else {
        nM = min(b, d.s_cnt[i]);
        const uint64_t *S = d.s_old + (size_t)i * d.s_cap;
        for (int t = tid; t < nM; t += T) {
            const uint64_t k = d.warm ? S[t] : S[t] & ~1ull;
            M[t] = k;
            if (!d.warm) mark_bit(seen, key_id(k));
        }
    }
    if (tid == 0) {
        s_nev = d.first && EV ? 1 : 0;
        s_end = 0;
    }
    __syncthreads();
    int nI = 0, nvis = 0, Kt = 2, ns = 0;
    int cM = 0, cI = 0;  // warp 0: everything before them is visited
    uint64_t tau = (nM >= b) ? (M[b - 1] | 1ull) : kEmpty;
    const int64_t limit = min(d.v_cap, a.iter_limit);

    // M <- top-b(M u I), I empty
    auto flush = [&]() {
        for (int t = tid; t < nM; t += T) {
            const uint64_t k = M[t];
            const int pos = t + lb_or1(I, nI, k | 1ull);
            if (pos < b) M2[pos] = k;
        }
        for (int t = tid; t < nI; t += T) {
            const uint64_t k = I[t];
            const int pos = t + lb_or1(M, nM, k | 1ull);
            if (pos < b) M2[pos] = k;
        }
        if (warp == 0) {
            const int pM = cM < nM ? cM + lb_or1(I, nI, M[cM] | 1ull) : 0x7fffffff;
            const int pI = cI < nI ? cI + lb_or1(M, nM, I[cI] | 1ull) : 0x7fffffff;
            cM = min(pM, pI);
            cI = 0;
        }
        __syncthreads();
        nM = min(b, nM + nI);
        if (warp == 0) cM = min(cM, nM);
        nI = 0;
        uint64_t *t = M;
        M = M2;
        M2 = t;
    };
    // the first n unvisited keys of L[c..nL) up to tau with their positions; c moves to the first (warp 0)
    auto pick = [&](const uint64_t *L, int nL, int &c, int n, uint64_t *ok, int *op) {
        int got = 0;
        for (int t0 = c; t0 < nL && got < n; t0 += 32) {
            const int t = t0 + lane;
            const uint64_t k = t < nL ? L[t] : kEmpty;
            const bool un = t < nL && !(k & 1ull);
            const unsigned m = __ballot_sync(0xffffffffu, un);
            if (got == 0) c = m ? t0 + __ffs(m) - 1 : min(t0 + 32, nL);
            const int r = got + __popc(m & lanemask_lt());
            if (un && r < n) {
                ok[r] = k;
                op[r] = t;
            }
            got = min(n, got + __popc(m));
            if ((__shfl_sync(0xffffffffu, k, 31) | 1ull) > tau) break;
        }
        return got;
    };

    for (int it = 0;; it ^= 1) {
        if (warp == 0) {
            if (ns > 0) {
                int j;
                tau = warp_kth_or1(M, nM, I, nI, b, &j);
                nI = j;
                cI = min(cI, nI);
            }
            // the next parents: the Kt smallest unvisited keys of the beam
            const int gM = pick(M, nM, cM, Kt, selk, selp);
            const int gI = pick(I, nI, cI, Kt, selk + CW, selp + CW);
            __syncwarp();
            const bool inM = lane < gM, inI = lane >= CW && lane < CW + gI;
            bool use = false;
            if (inM || inI) {
                const uint64_t k = selk[lane];
                const uint64_t *o = inM ? selk + CW : selk;
                const int no = inM ? gI : gM;
                int r = inM ? lane : lane - CW;
                for (int t = 0; t < no; t++) r += o[t] < k;
                use = r < Kt && (k | 1ull) <= tau;
                if (use) {
                    pkey[r] = k;
                    ppos[r] = inM ? selp[lane] : -1 - selp[lane];
                }
            }
            int K = __popc(__ballot_sync(0xffffffffu, use));
            __syncwarp();
            if (a.use_es && K > 0) {
                uint64_t mn = M[0] | 1ull;
                if (nI > 0 && (I[0] | 1ull) < mn) mn = I[0] | 1ull;
                const bool fire = lane < K && key_dk(mn) > rks && nvis + lane >= a.es_vl && key_dk(pkey[lane & (CW - 1)]) > ek;
                const unsigned m = __ballot_sync(0xffffffffu, fire);
                if (m) K = __ffs(m) - 1;
                if (K == 0 && lane == 0) s_end = 1;
            }
            if (K > 0 && nvis + K > limit) {
                K = (int)(limit - nvis);
                if (K == 0 && lane == 0) {
                    if (nvis >= a.iter_limit) atomicExch(a.error, 2);
                    else s_end = 2;
                }
            }
            if (lane == 0) {
                s_K = K;
                s_tau = tau;
                s_nI = nI;
                s_ns[it] = 0;
            }
        }
        __syncthreads();
        const int K = s_K;
        if (K == 0) break;
        tau = s_tau;
        nI = s_nI;
        // a group of warps per parent, each a part of its row: the unseen neighbours and their distances
        const int lg = K <= 1 ? 0 : 32 - __clz(K - 1);   // parents rounded up to 2^lg
        const int G = CW >> lg, par = warp / G;
        int nc = 0;
        if (par < K) {
            const int part = (R + G - 1) / G, e1 = min(R, (warp % G + 1) * part);
            const uint32_t *row = a.adj + (size_t)key_id(pkey[par]) * R;
            for (int e0 = (warp % G) * part; e0 < e1; e0 += 32) {
                const int e = e0 + lane;
                const uint32_t j = e < e1 ? __ldg(row + e) : kSent;
                const bool v = j < (uint32_t)a.n && !((__ldcg(seen + (j >> 5)) >> (j & 31)) & 1u);
                const unsigned m = __ballot_sync(0xffffffffu, v);
                if (v) cid[nc + __popc(m & lanemask_lt())] = j;
                nc += __popc(m);
            }
            __syncwarp();
            uint32_t mn = 0xffffffffu;
            if (nc > 0) {
                if constexpr (LP) eval_candidates_lp<DT, DT == DT_FP8 ? 4 : 8>(a, qf, qn2, cid, nc, ckey);
                else eval_candidates<DT, CPL, UN>(a, q, cid, nc, ckey);
                __syncwarp();
                for (int c = lane; c < nc; c += 32) mn = min(mn, key_dk(ckey[c]));
                mn = __reduce_min_sync(0xffffffffu, mn);
            }
            if (lane == 0) mind[warp] = mn;
        }
        __syncthreads();
        int nk = 1;
        for (uint32_t mn = 0xffffffffu; nk < K; nk++) {
            for (int w = (nk - 1) * G; w < nk * G; w++) mn = min(mn, mind[w]);
            if (mn <= key_dk(pkey[nk])) break;
        }
        // V <- V u the first nk parents
        if (warp == 0 && lane < nk) {
            const int pos = ppos[lane];
            V[nvis + lane] = pkey[lane] & ~1ull;
            if (pos >= 0) M[pos] |= 1ull;
            else I[-1 - pos] |= 1ull;
        }
        if (par < nk) {
            for (int c0 = 0; c0 < nc; c0 += 32) {
                const int c = c0 + lane;
                const uint64_t k = c < nc ? ckey[c] : kEmpty;
                const bool v = c < nc && mark_bit(seen, key_id(k));
                const unsigned m = __ballot_sync(0xffffffffu, v);
                if (EV && m) {
                    int at = 0;
                    if (lane == 0) at = atomicAdd(&s_nev, __popc(m));
                    at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & lanemask_lt());
                    if (v && at < d.ev_cap) EV[at] = k;
                }
                const bool keep = v && (k | 1ull) < tau;
                const unsigned mk = __ballot_sync(0xffffffffu, keep);
                if (mk) {
                    int at = 0;
                    if (lane == 0) at = atomicAdd(&s_ns[it], __popc(mk));
                    at = __shfl_sync(0xffffffffu, at, 0);
                    if (keep) skey[at + __popc(mk & lanemask_lt())] = k;
                }
            }
        }
        __syncthreads();
        nvis += nk;
        Kt = nk == K ? min(CW, 2 * nk) : nk + 1;
        if (EV && s_nev > d.ev_cap) {
            if (tid == 0) s_end = 2;
            break;
        }
        ns = s_ns[it];
        if (ns == 0) continue;
        if (nI + ns > ki) flush();
        for (int c = tid; c < ns; c += T) {  // sort by rank: distinct keys
            const uint64_t k = skey[c];
            int r = 0;
            for (int t = 0; t < ns; t++) r += skey[t] < k;
            ckeys[r] = k;
        }
        __syncthreads();
        // I <- I u survivors
        for (int t = tid; t < nI; t += T) {
            const uint64_t k = I[t];
            I2[t + lb_or1(ckeys, ns, k | 1ull)] = k;
        }
        for (int t = tid; t < ns; t += T) {
            const uint64_t k = ckeys[t];
            I2[t + lb_or1(I, nI, k | 1ull)] = k;
        }
        if (warp == 0) cI = min(cI, lb_or1(I, nI, ckeys[0] | 1ull));
        __syncthreads();
        nI += ns;
        uint64_t *t = I;
        I = I2;
        I2 = t;
    }
    __syncthreads();
    if (s_nI > 0) {
        nI = s_nI;
        flush();
        __syncthreads();
    }
    const bool stopped = s_end == 1, overflow = s_end == 2;
    // N = {n in B : d <= r}, a prefix of M
    int cnt = 0;
    for (int hi = nM; cnt < hi;) {
        const int mid = (cnt + hi) >> 1;
        if (key_dk(M[mid]) <= rks) cnt = mid + 1;
        else hi = mid;
    }
    if constexpr (LP) {
        __syncthreads();
        if (warp == 0) {
            const int c = exact_filter_sort<CPL, UN>(a, qi, M, cnt, rk, cid, ckey, R);
            if (lane == 0) s_cnt = c;
        }
        __syncthreads();
        cnt = s_cnt;
    }
    const bool cont = !stopped && !overflow && cnt == b && !d.last;
    if (!cont) {
        // finished: append N to the result items
        if (tid == 0) s_base = cnt > 0 ? atomicAdd(d.tail, (unsigned long long)cnt) : 0ull;
        __syncthreads();
        const unsigned long long base = s_base, cap = (unsigned long long)d.cap;
        const int fit = base >= cap ? 0 : (int)min((unsigned long long)cnt, cap - base);
        for (int t = tid; t < fit; t += T) {
            d.item_key[base + t] = M[t] & ~1ull;
            d.item_slot[base + t] = slot;
        }
        if (tid == 0) {
            d.slot_count[slot] = fit;
            d.slot_trunc[slot] = (fit < cnt || overflow || (d.last && cnt == b && !stopped)) ? 1 : 0;
        }
    }
    if (tid == 0) {
        d.status[i] = cont ? 1 : 0;
        d.nv[i] = nvis;
        if (d.nev) d.nev[i] = s_nev;
    }
}

// CTA per continuing slot: S_new <- the s_cap_new smallest distinct keys of S_old u V.
__global__ void __launch_bounds__(1024) supdate_kernel(DoublingSUpdate u, int smem_cap) {
    extern __shared__ __align__(16) uint8_t smem_raw[];
    uint64_t *sk = reinterpret_cast<uint64_t *>(smem_raw);
    __shared__ int wsum[32];
    for (int j = blockIdx.x; j < u.nc; j += gridDim.x) {
        const int i = u.cont[j];
        const int ns = u.first ? 0 : u.s_cnt_old[i];
        const int ne = u.warm ? u.nev[i] : 0;
        const int nv = u.nv[i];
        const int m = ns + ne + nv;
        uint64_t *a = m <= smem_cap ? sk : u.tmp + (size_t)j * (u.s_cap_old + (u.warm ? u.ev_cap : 0) + u.v_cap);
        const uint64_t *S = u.s_old + (size_t)i * u.s_cap_old;
        const uint64_t *EV = u.warm ? u.ev + (size_t)i * u.ev_cap : nullptr;
        const uint64_t *V = u.v + (size_t)i * u.v_cap;
        for (int t = threadIdx.x; t < m; t += blockDim.x) {
            if (!u.warm) a[t] = (t < ns ? S[t] : V[t - ns]) & ~1ull;
            // warm restart: E's keys keep their visited bits, this round's visits get theirs
            else a[t] = t < ns ? S[t] : (t < ns + ne ? EV[t - ns] & ~1ull : V[t - ns - ne] | 1ull);
        }
        __syncthreads();
        // bitonic sort with flip stages (min to the lower index; virtual +inf padding)
        int P = 1;
        while (P < m) P <<= 1;
        for (int k = 2; k <= P; k <<= 1) {
            for (int jj = k >> 1; jj > 0; jj >>= 1) {
                const int lj = __ffs(jj) - 1;  // powers of two: shifts and masks
                for (int t = threadIdx.x; t < P / 2; t += blockDim.x) {
                    const int off = t & (jj - 1);
                    const int lo = ((t >> lj) << (lj + 1)) + off;
                    const int hi = (jj == (k >> 1)) ? lo - off + (k - 1 - off) : lo + jj;
                    if (hi < m) {
                        uint64_t x = a[lo], y = a[hi];
                        if (y < x) { a[lo] = y; a[hi] = x; }
                    }
                }
                __syncthreads();
            }
        }
        // drop repeated keys (S and V share ids), keep the first s_cap_new distinct ones; warm restart: of the
        // copies of a key (with and without the visited bit) keep the last, which carries the bit if any does
        uint64_t *out = u.s_new + (size_t)j * u.s_cap_new;
        int carry = 0;
        for (int b0 = 0; b0 < m; b0 += blockDim.x) {
            int t = b0 + threadIdx.x;
            int keep;
            if (!u.warm) keep = (t < m && (t == 0 || a[t] != a[t - 1])) ? 1 : 0;
            else keep = (t < m && (t == m - 1 || (a[t] | 1ull) != (a[t + 1] | 1ull))) ? 1 : 0;
            unsigned bm = __ballot_sync(0xffffffffu, keep);
            int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
            int pre = __popc(bm & ((1u << lane) - 1));
            if (lane == 0) wsum[w] = __popc(bm);
            __syncthreads();
            int wo = 0;
            for (int x = 0; x < w; x++) wo += wsum[x];
            int tot = 0;
            for (int x = 0; x < (int)(blockDim.x >> 5); x++) tot += wsum[x];
            int pos = carry + wo + pre;
            if (keep && pos < u.s_cap_new) out[pos] = a[t];
            carry += tot;
            __syncthreads();
        }
        if (threadIdx.x == 0) u.s_cnt_new[j] = carry < u.s_cap_new ? carry : (int)u.s_cap_new;
        __syncthreads();
    }
}

__global__ void zero_words_kernel(uint32_t *p, int64_t n) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) p[t] = 0;
}

// Two CTAs of 256 threads (111 registers) fit an SM: up to two waves of them a round goes by CTA.  With more active
// queries a warp each fills the chip, and the evaluations made for nothing would cost throughput.  At the limit the
// phase is still 2.1 times (fp32 2 KB, R = 128: 32.0 -> 15.1 ms) to 2.8 times faster (u8 128 B, R = 128: 17.1 -> 6.2; fp32
// 800 B, R = 64: 21.0 -> 7.5); at 40 queries 2.4 to 3.0 times.  Exact counters
// (stats) are kept by the warp form only: rr_query_stats.evals is what was evaluated, and the lookahead evaluates more.
constexpr int kCtaRounds = 608;

template <int DT, int CPL>
rr_status round_t(const DoublingRound &d, cudaStream_t st) {
    if (d.na <= kCtaRounds && !d.s.stats) {
        note_form(kFormRoundCta);
        const size_t smem = round_cta_smem_bytes(d.s.R);
        auto k = round_cta_kernel<DT, CPL>;
        if (rr_status e = allow_smem((const void *)k, smem)) return e;
        k<<<(unsigned)d.na, 32 * CW, smem, st>>>(d);
        RR_CUDA(cudaGetLastError());
        note_launch();
        return RR_OK;
    }
    note_form(kFormRoundWarp);
    const int wpc = 4;
    size_t smem = (size_t)wpc * round_smem_bytes(d.s.R);
    auto k = round_kernel<DT, CPL>;
    if (rr_status e = allow_smem((const void *)k, smem)) return e;
    k<<<(unsigned)((d.na + wpc - 1) / wpc), 32 * wpc, smem, st>>>(d);
    RR_CUDA(cudaGetLastError());
    note_launch();
    return RR_OK;
}

}  // namespace

rr_status launch_doubling_round(const DoublingRound &d, cudaStream_t st, int dtype_code) {
    if (d.na <= 0) return RR_OK;
    const int cpl = (d.s.row_chunks + 31) / 32;
    switch (dtype_code) {
        case DT_U8: return round_t<DT_U8, 1>(d, st);
        case DT_I8: return round_t<DT_I8, 1>(d, st);
        case DT_F32:
            if (d.s.prec == RR_PREC_BF16) return cpl <= 2 ? round_t<DT_BF16, 2>(d, st) : round_t<DT_BF16, 4>(d, st);
            if (d.s.prec == RR_PREC_FP8) return cpl <= 2 ? round_t<DT_FP8, 2>(d, st) : round_t<DT_FP8, 4>(d, st);
            if (cpl <= 1) return round_t<DT_F32, 1>(d, st);
            if (cpl <= 2) return round_t<DT_F32, 2>(d, st);
            return round_t<DT_F32, 4>(d, st);
    }
    set_error("doubling phase: unsupported element type %d", dtype_code);
    return RR_EINVAL;
}

rr_status launch_doubling_supdate(const DoublingSUpdate &u, cudaStream_t st) {
    if (u.nc <= 0) return RR_OK;
    const int smem_cap = 16384;
    size_t smem = (size_t)smem_cap * 8;
    if (rr_status e = allow_smem((const void *)supdate_kernel, smem)) return e;
    int blocks = u.nc < 152 * 2 ? u.nc : 152 * 2;
    supdate_kernel<<<blocks, 1024, smem, st>>>(u, smem_cap);
    RR_CUDA(cudaGetLastError());
    note_launch();
    return RR_OK;
}

rr_status launch_zero_words(uint32_t *p, int64_t n, cudaStream_t st) {
    if (n <= 0) return RR_OK;
    int64_t blocks = (n + 255) / 256;
    if (blocks > 152 * 32) blocks = 152 * 32;
    zero_words_kernel<<<(unsigned)blocks, 256, 0, st>>>(p, n);
    RR_CUDA(cudaGetLastError());
    note_launch();
    return RR_OK;
}

}  // namespace rr
