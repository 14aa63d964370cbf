// qm_weighted.cuh -- Eqs. (8)-(9) on weighted graphs (included by qm_kernels.cu).
//
// The paper defines Q and Qds for unweighted graphs and notes for the
// weighted case that the densities d_c and d_ci,cj keep the unweighted edge
// counts (so that they stay at most 1) while the other edge amounts become
// weight sums:
//   Q_w   = sum_c [ W_c^in / W - ((2 W_c^in + W_c^out) / (2W))^2 ]
//   Qds_w = sum_ci [ W_ci^in / W d_ci - ((2 W_ci^in + W_ci^out) / (2W) d_ci)^2
//                    - sum_{cj != ci} W_ci,cj / (2W) d_ci,cj ]
// Weights are float32 (0 or in [2^-20, 2^20)); each is an exact fixed-point
// integer w * 2^43, so every weight sum below is exact:
//   - k_rows<true> sums each community's intra-arc weights (2 W_c^in) and
//     cut-arc weights (W_c^out) into three-word integers, and packs the cut
//     arcs' weights beside their labels;
//   - k_count_w_tab and k_count_w_big count each community's run in a
//     shared-memory table (|E_ci,cj| for every neighbour cj) and then, in a
//     second pass over the run, add for every cut arc (weight w, neighbour cj)
//     the exact product w * |E_ci,cj| * Rcp_cj, so that
//     P_i = sum_j W_ij |E_ij| / |c_j| is a 256-bit integer (scale 2^171);
//   - k_score_terms_w forms the FP64 terms of each community once from these
//     integers and adds them in fixed point (Q_w into its own accumulator).
// The six measures of Sec. II-B.3 keep their unweighted counts.
//
// Included inside namespace qm of qm_kernels.cu, after the helpers it uses.

struct U256 {
    unsigned long long w[4];
};

__device__ __forceinline__ void u256_zero(U256 &a) { a.w[0] = a.w[1] = a.w[2] = a.w[3] = 0ull; }

__device__ __forceinline__ void u256_add(U256 &a, const U256 &b)
{
    unsigned long long c = 0ull;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const unsigned long long s = a.w[k] + b.w[k];
        const unsigned long long c1 = s < a.w[k] ? 1ull : 0ull;
        const unsigned long long t = s + c;
        const unsigned long long c2 = t < s ? 1ull : 0ull;
        a.w[k] = t;
        c = c1 + c2;
    }
}

// a += x * r for x < 2^96 and a 128-bit reciprocal r (the product is below 2^224).
__device__ __forceinline__ void u256_mac(U256 &a, u128 x, const Rcp &r)
{
    const unsigned long long x0 = (unsigned long long)x, x1 = (unsigned long long)(x >> 64);
    const unsigned long long r0 = r.lo, r1 = r.hi;
    const u128 p00 = (u128)x0 * r0, p01 = (u128)x0 * r1, p10 = (u128)x1 * r0, p11 = (u128)x1 * r1;
    U256 p;
    p.w[0] = (unsigned long long)p00;
    u128 t = (p00 >> 64) + (u128)(unsigned long long)p01 + (u128)(unsigned long long)p10;
    p.w[1] = (unsigned long long)t;
    t = (t >> 64) + (p01 >> 64) + (p10 >> 64) + (u128)(unsigned long long)p11;
    p.w[2] = (unsigned long long)t;
    p.w[3] = (unsigned long long)((t >> 64) + (p11 >> 64));
    u256_add(a, p);
}

__device__ __forceinline__ double u256_to_double(const U256 &a)
{
    double r = (double)a.w[3];
    r = __dadd_rn(__dmul_rn(r, 18446744073709551616.0), (double)a.w[2]);
    r = __dadd_rn(__dmul_rn(r, 18446744073709551616.0), (double)a.w[1]);
    r = __dadd_rn(__dmul_rn(r, 18446744073709551616.0), (double)a.w[0]);
    return r;  // a, rounded (its value times 2^0)
}

// Count of `key` in the table (0 when absent).
__device__ __forceinline__ unsigned long long tab_count(const SmemTable &t, unsigned key)
{
    const unsigned long long tag = (unsigned long long)(key + 1u) << 32;
    unsigned h = tab_hash(key, t.cap);
    for (int probe = 0; probe < t.cap; ++probe) {
        if (!QM_CHK(h, t.cap, 11)) return 0ull;
        const unsigned long long s = ((volatile unsigned long long *)t.slot)[h];
        if ((s & 0xFFFFFFFF00000000ull) == tag) return s & 0xFFFFFFFFull;
        if (s == 0ull) return 0ull;
        h = (h + 1u == (unsigned)t.cap) ? 0u : h + 1u;
    }
    return 0ull;
}

// Block totals of (slots, cnt2, P) delivered to thread 0 (6 words per warp in red).
__device__ __forceinline__ void group_totals_w(unsigned long long &slots, unsigned long long &cnt2, U256 &P,
                                               unsigned long long *red)
{
    slots = warp_sum_u64(slots);
    cnt2 = warp_sum_u64(cnt2);
    for (int d = 16; d > 0; d >>= 1) {
        U256 o;
#pragma unroll
        for (int k = 0; k < 4; ++k) o.w[k] = __shfl_down_sync(0xffffffffu, P.w[k], d);
        u256_add(P, o);
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    block_sync();
    if (lane == 0) {
        red[6 * wid] = slots;
        red[6 * wid + 1] = cnt2;
#pragma unroll
        for (int k = 0; k < 4; ++k) red[6 * wid + 2 + k] = P.w[k];
    }
    block_sync();
    if (threadIdx.x == 0)
        for (int w = 1; w < nw; ++w) {
            slots += red[6 * w];
            cnt2 += red[6 * w + 1];
            U256 o;
#pragma unroll
            for (int k = 0; k < 4; ++k) o.w[k] = red[6 * w + 2 + k];
            u256_add(P, o);
        }
}

// Counts community c's run (entries nbr[a0 .. a0 + m), weights nbrw[...]) with
// the whole block, then adds every entry's weighted pair share.  Runs larger
// than the table split their keys into R hash classes (one pass per class);
// an overflowing pass doubles R.  Writes rec[c] (REC_* words; the unweighted
// pair sum is not formed) and recw[c] = P_c (256-bit).
__device__ __forceinline__ void count_run_weighted(const CountCtx &x, const float *nbrw, unsigned long long *recw,
                                                   int c, unsigned a0, unsigned m, unsigned vol,
                                                   const SmemTable &tab, int tid, int T, unsigned long long *red)
{
    const int *src = x.nbr + a0;
    const float *wsrc = nbrw + a0;
    const unsigned cap_keys = (unsigned)tab.max_used;
    unsigned R = m <= cap_keys ? 1u
                               : (unsigned)min((unsigned long long)R_MAX,
                                               (5ull * m + 4ull * cap_keys - 1) / (4ull * cap_keys));
    for (;;) {
        unsigned long long slots = 0, cnt2 = 0;
        U256 P;
        u256_zero(P);
        bool ok = true;
        for (unsigned r = 0; r < R && ok; ++r) {
            for (unsigned e = tid; e < m; e += T) {
                const int lv = __ldcg(&src[e]);
                if (!QM_CHK(lv, x.K, 6)) continue;
                if (R == 1 || tab_split((unsigned)lv, R) == r) tab_insert(tab, (unsigned)lv);
            }
            block_sync();
            if (*(volatile int *)tab.overflow) {
                ok = false;
                break;
            }
            for (unsigned e = tid; e < m; e += T) {
                const int lv = __ldcg(&src[e]);
                if (!QM_CHK(lv, x.K, 6)) continue;
                if (R > 1 && tab_split((unsigned)lv, R) != r) continue;
                const unsigned long long cnt = tab_count(tab, (unsigned)lv);
                const u128 q = (u128)w_fixed(__ldcg(&wsrc[e])) * (u128)cnt;
                u256_mac(P, q, ld_rcp(&x.recip[lv]));
            }
            block_sync();
            tab_drain(tab, tid, T, [&](int key, long long cnt) {
                if (key < c) return;  // each unordered pair counted once, by its smaller id
                ++slots;
                cnt2 += (unsigned long long)cnt * (unsigned long long)cnt;
            });
            block_sync();
            if (tid == 0) *tab.n_used = 0;
            block_sync();
        }
        if (!ok) {
            tab_wipe(tab, tid, T);
            block_sync();
            if (tid == 0) { *tab.n_used = 0; *tab.overflow = 0; }
            block_sync();
            const unsigned nr = R * 2u;
            if (nr > R_MAX) {
                if (tid == 0) atomicOr(x.err, 2);
                return;
            }
            R = nr;
            continue;
        }
        group_totals_w(slots, cnt2, P, red);
        if (tid == 0) {
            unsigned long long *rc = x.rec + (size_t)c * REC_WORDS;
            rc[REC_SAME] = (unsigned long long)(vol - m);
            rc[REC_VOL] = (unsigned long long)vol;
            rc[REC_SLOTS] = slots;
            rc[REC_CNT2] = cnt2;
            rc[REC_INNER_LO] = 0ull;
            rc[REC_INNER_HI] = 0ull;
            rc[REC_FULL_LO] = 0ull;
            rc[REC_FULL_HI] = 0ull;
#pragma unroll
            for (int k = 0; k < 4; ++k) recw[(size_t)c * 4 + k] = P.w[k];
        }
        block_sync();
        return;
    }
}

// a += x * r for x < 2^64.
__device__ __forceinline__ void u256_mac64(U256 &a, unsigned long long x, const Rcp &r)
{
    const u128 p0 = (u128)x * r.lo, p1 = (u128)x * r.hi;
    const u128 t = p1 + (unsigned long long)(p0 >> 64);  // below 2^128: (2^64 - 1)^2 + 2^64 - 1
    asm("add.cc.u64 %0, %0, %4;\n\taddc.cc.u64 %1, %1, %5;\n\taddc.cc.u64 %2, %2, %6;\n\taddc.u64 %3, %3, 0;"
        : "+l"(a.w[0]), "+l"(a.w[1]), "+l"(a.w[2]), "+l"(a.w[3])
        : "l"((unsigned long long)p0), "l"((unsigned long long)t), "l"((unsigned long long)(t >> 64)));
}

// Warp total of a 256-bit sum (valid in every lane): ten 27-bit chunks, each
// added by one redux.
__device__ __forceinline__ U256 ct_warp_sum256(const U256 &a)
{
    U256 r;
    u256_zero(r);
#pragma unroll
    for (int k = 0; k < 10; ++k) {
        const int at = 27 * k, w = at / 64, s = at % 64;
        unsigned long long v = a.w[w] >> s;
        if (s > 37 && w < 3) v |= a.w[w + 1] << (64 - s);
        const unsigned long long sum = __reduce_add_sync(0xffffffffu, (unsigned)v & ((1u << 27) - 1u));
        U256 t;
        u256_zero(t);
        t.w[w] = sum << s;
        if (s > 32 && w < 3) t.w[w + 1] = sum >> (64 - s);
        u256_add(r, t);
    }
    return r;
}

// Counts community h.c's run (labels nbr[a0 ..), weights nbrw[a0 ..), m entries)
// with a group of GS threads and the one-word tables of qm_count.cuh: every
// label's occurrences in a first pass over the run, then every entry's exact
// share w |E_cj| Rcp_j in a second (the same integer whatever the order).
// Bound by the instructions of the two passes.  6.5*10^7 cut arcs of 10^7
// nodes: 2.71 ms for whole blocks on 64-bit tables with a pass to clear them,
// 1.23 ms so (k_count_w_tab 0.59, k_count_w_big 0.64).
template <int GS>
__device__ __forceinline__ void ct_count_run_weighted(const CountCtx &x, const RunHdr &h, const float *nbrw,
                                                      unsigned long long *recw, unsigned *slot, int cb, int gtid,
                                                      unsigned *late, unsigned long long *red)
{
    constexpr unsigned ALL = 0xffffffffu;
    const int m = (int)h.m, c = h.c, lane = threadIdx.x & 31;
    const int *src = x.nbr + h.a0;
    const float *wsrc = nbrw + h.a0;
    const unsigned lt = (1u << lane) - 1u, one = 1u << cb;
    const unsigned lg = ct_slots_log2(h.m), mask = (1u << lg) - 1u, shift = 32u - lg;
    unsigned counts[3] = {0u, 0u, 0u};  // above c: repeats, twice the occurrences before them, entries
    unsigned nl = 0;
    auto follow = [&](unsigned n) {
        nl -= n;
        const unsigned key = (unsigned)lane < n ? late[nl + lane] : 0u;
        const unsigned before = ct_follow(slot, key, mask, shift, cb);
        if (before && (int)(key - 1u) > c) {
            counts[0] += 1u;
            counts[1] += 2u * before;
        }
        __syncwarp();
    };
    for (int e0 = gtid & ~31; e0 < m; e0 += GS * CT_UNROLL) {
        int lv[CT_UNROLL];
        unsigned cur[CT_UNROLL];
#pragma unroll
        for (int k = 0; k < CT_UNROLL; ++k) {
            const int e = e0 + lane + GS * k;
            lv[k] = e < m ? __ldg(&src[e]) : -1;
            if (lv[k] >= 0 && !QM_CHK(lv[k], x.K, 6)) lv[k] = -1;
            counts[2] += lv[k] > c ? 1u : 0u;
        }
#pragma unroll
        for (int k = 0; k < CT_UNROLL; ++k) {
            const unsigned hs = ((unsigned)lv[k] * 0x9E3779B1u) >> shift;
            cur[k] = lv[k] >= 0 ? atomicCAS(&slot[hs], 0u, (unsigned)lv[k] * one + one) : 0u;
        }
#pragma unroll
        for (int k = 0; k < CT_UNROLL; ++k) {
            const unsigned taken = __ballot_sync(ALL, cur[k] != 0u);
            if (cur[k] != 0u) late[nl + __popc(taken & lt)] = (unsigned)lv[k] + 1u;
            nl += __popc(taken);
        }
        __syncwarp();
        while (nl >= 32u) follow(32u);
    }
    if (nl) follow(nl);
    ct_sync<GS>();
    U256 P;
    u256_zero(P);
    for (int e0 = gtid & ~31; e0 < m; e0 += GS * CT_UNROLL) {
        int lv[CT_UNROLL];
        float wv[CT_UNROLL];
        unsigned cnt[CT_UNROLL], hs[CT_UNROLL];
        Rcp rj[CT_UNROLL];
#pragma unroll
        for (int k = 0; k < CT_UNROLL; ++k) {
            const int e = e0 + lane + GS * k;
            lv[k] = e < m ? __ldg(&src[e]) : -1;
            wv[k] = e < m ? __ldcs(&wsrc[e]) : 0.0f;
            if (lv[k] >= 0 && !QM_CHK(lv[k], x.K, 6)) lv[k] = -1;
            rj[k] = Rcp{0ull, 0ull};
            if (lv[k] >= 0) rj[k] = ld_rcp(&x.recip[lv[k]]);
            hs[k] = ((unsigned)lv[k] * 0x9E3779B1u) >> shift;
            cnt[k] = 0u;
        }
        // every key is in the table: each lane steps on until it meets its own
        for (unsigned step = 0; step <= mask; ++step) {
            bool pend = false;
#pragma unroll
            for (int k = 0; k < CT_UNROLL; ++k) {
                if (lv[k] < 0 || cnt[k]) continue;
                const unsigned v = ((volatile unsigned *)slot)[hs[k]];
                if ((v >> cb) == (unsigned)lv[k] + 1u) cnt[k] = (v & (one - 1u)) + 1u;
                else pend = true;
                hs[k] = (hs[k] + 1u) & mask;
            }
            if (!__any_sync(ALL, pend)) break;
        }
#pragma unroll
        for (int k = 0; k < CT_UNROLL; ++k) {
            const u128 q = (u128)w_fixed(wv[k]) * cnt[k];  // 0 where there is no entry
            const bool wide = (unsigned long long)(q >> 64) != 0ull;
            u256_mac64(P, wide ? 0ull : (unsigned long long)q, rj[k]);
            if (__any_sync(ALL, wide)) {
                if (wide) u256_mac(P, q, rj[k]);
                __syncwarp();
            }
        }
    }
    ct_sync<GS>();
    for (unsigned i = (unsigned)gtid; i < (1u << lg) / 4u; i += (unsigned)GS)
        reinterpret_cast<uint4 *>(slot)[i] = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int k = 0; k < 3; ++k) counts[k] = __reduce_add_sync(ALL, counts[k]);
    P = ct_warp_sum256(P);
    if (GS > 32) {
        const int wid = threadIdx.x >> 5;
        if (lane == 0) {
            unsigned long long *r = red + 6 * wid;
            r[0] = ((unsigned long long)counts[2] << 32) | counts[0];
            r[1] = counts[1];
#pragma unroll
            for (int k = 0; k < 4; ++k) r[2 + k] = P.w[k];
        }
        ct_sync<GS>();
        if (threadIdx.x == 0)
            for (int v = 1; v < GS / 32; ++v) {
                const unsigned long long *r = red + 6 * v;
                counts[0] += (unsigned)r[0];
                counts[2] += (unsigned)(r[0] >> 32);
                counts[1] += (unsigned)r[1];
                u256_add(P, U256{{r[2], r[3], r[4], r[5]}});
            }
    }
    if (gtid == 0) {
        unsigned long long *rc = x.rec + (size_t)c * REC_WORDS;
        rc[REC_SAME] = (unsigned long long)(h.vol - h.m);
        rc[REC_VOL] = (unsigned long long)h.vol;
        rc[REC_SLOTS] = (unsigned long long)(counts[2] - counts[0]);
        rc[REC_CNT2] = (unsigned long long)counts[2] + counts[1];
        rc[REC_INNER_LO] = rc[REC_INNER_HI] = rc[REC_FULL_LO] = rc[REC_FULL_HI] = 0ull;
#pragma unroll
        for (int k = 0; k < 4; ++k) recw[(size_t)c * 4 + k] = P.w[k];
    }
    ct_sync<GS>();
}

struct CountWArgs {
    CountCtx x;
    const float *nbrw;
    unsigned long long *recw;
    const RunHdr *big, *small, *lng, *mid;
    int *counters;
    const int *status;
    int cb;
    SmemPlan plan;  // hash-class tables of k_count_w_big
};

// As k_count_tab.  (The block's second pass re-reads the run from L1 / L2.)
__global__ void __launch_bounds__(CT_THREADS, 6) k_count_w_tab(CountWArgs a)
{
    __shared__ __align__(16) unsigned slot[CT_WORDS];
    __shared__ unsigned late[CT_THREADS / 32][CT_LATE];
    __shared__ unsigned long long red[6 * (CT_THREADS / 32)];
    __shared__ int s_i;
    if (*a.status) return;
    constexpr int W = CT_THREADS / 32;
    const int tid = threadIdx.x, wid = tid >> 5, lane = tid & 31;
    for (int i = tid; i < CT_WORDS / 4; i += CT_THREADS)
        reinterpret_cast<uint4 *>(slot)[i] = make_uint4(0u, 0u, 0u, 0u);
    const int nmid = a.counters[C_MID_COUNT];
    for (;;) {
        if (tid == 0) s_i = atomicAdd(&a.counters[C_MID_NEXT], 1);
        block_sync();
        const int i = s_i;
        if (i >= nmid) break;
        ct_count_run_weighted<CT_THREADS>(a.x, a.mid[i], a.nbrw, a.recw, slot, a.cb, tid, late[wid], red);
    }
    const int nsmall = a.counters[C_SMALL_COUNT];
    const int chunk = claim_chunk(nsmall, (long long)gridDim.x * W);
    unsigned *const ws = slot + wid * (CT_WORDS / W);
    for (;;) {
        int base = 0;
        if (lane == 0) base = atomicAdd(&a.counters[C_SMALL_NEXT], chunk);
        base = __shfl_sync(0xffffffffu, base, 0);
        if (base >= nsmall) break;
        const int top = min(nsmall, base + chunk);
        for (int i = base; i < top; ++i)
            ct_count_run_weighted<32>(a.x, a.small[i], a.nbrw, a.recw, ws, a.cb, lane, late[wid], red);
    }
}

// The longer runs: one table in the block's shared memory up to CB_FILL_LONG
// entries (and below 2^cb), then hash classes.
__global__ void __launch_bounds__(CB_THREADS, 2) k_count_w_big(CountWArgs a)
{
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ unsigned late[CB_THREADS / 32][CT_LATE];
    __shared__ unsigned long long red[6 * (CB_THREADS / 32)];
    if (block_stopped(a.status)) return;
    const int nbig = a.counters[C_BIG_COUNT], nlong = a.counters[C_LONG_COUNT], tid = threadIdx.x;
    const int G = gridDim.x, b = blockIdx.x;
    if (b >= nbig && b >= nlong) return;
    unsigned *slot = (unsigned *)sm;
    for (int i = tid; i < CB_WORDS_LONG / 4; i += CB_THREADS)
        reinterpret_cast<uint4 *>(slot)[i] = make_uint4(0u, 0u, 0u, 0u);
    block_sync();
    for (int i = b; i < nbig; i += G)
        ct_count_run_weighted<CB_THREADS>(a.x, a.big[i], a.nbrw, a.recw, slot, a.cb, tid, late[tid >> 5], red);
    if (b >= nlong) return;
    const SmemPlan &p = a.plan;
    int *ctl = (int *)(sm + p.ctl_off);
    unsigned long long *lslot = (unsigned long long *)(sm + p.slot_off);
    int *used = (int *)(sm + p.used_off);
    for (int i = tid; i < p.cap; i += CB_THREADS) lslot[i] = 0ull;
    if (tid < 2) ctl[tid] = 0;
    block_sync();
    const SmemTable tb{lslot, used, &ctl[0], &ctl[1], p.cap, p.max_used};
    for (int i = b; i < nlong; i += G) {
        const RunHdr h = a.lng[i];
        count_run_weighted(a.x, a.nbrw, a.recw, h.c, h.a0, h.m, h.vol, tb, tid, CB_THREADS,
                           (unsigned long long *)(sm + p.red_off));
    }
}

// FP64 terms of every owned community from its integers (weighted Eqs. 8-9,
// unweighted Sec. II-B.3), added in fixed point; Q_w goes to GS_QW.
__global__ void k_score_terms_w(const unsigned long long *cv, const unsigned long long *rec, const unsigned long long *recw,
                                const unsigned long long *wl, int K, long long E, unsigned long long w_lo,
                                unsigned long long w_hi, PerCommDev pc, unsigned long long *g, const int *status,
                                Shard own, ScoreOut o)
{
    if (*status) return;
    ScoreAcc acc;
    score_acc_zero(acc);
    i128 qw = 0;
    const double W2 = __dmul_rn(2.0, u128_to_double(((u128)w_hi << 64) | (u128)w_lo));  // 2W * 2^43
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < K; c += gridDim.x * blockDim.x) {
        const long long size = (long long)(cv[c] >> VOL_BITS);
        if (size == 0 || !own.owns(c)) continue;
        const unsigned long long *rc = rec + (size_t)c * REC_WORDS;
        const unsigned long long same = rc[REC_SAME], vol = rc[REC_VOL];
        const long long ein = (long long)(same / 2), eout = (long long)(vol - same);
        double qs_unweighted, dens, contr, expn, cond;
        community_terms(ein, eout, size, E, qs_unweighted, dens, contr, expn, cond);
        const i128 win2 = wsum_get(wl + (size_t)c * 6), wout = wsum_get(wl + (size_t)c * 6 + 3);
        const double fin = __ddiv_rn(i128_to_double(win2), W2);          // W_c^in / W
        const double fvol = __ddiv_rn(i128_to_double(win2 + wout), W2);  // (2 W_c^in + W_c^out) / (2W)
        const double qwt = __dsub_rn(fin, __dmul_rn(fvol, fvol));
        const double t1 = __dmul_rn(fin, dens), t2 = __dmul_rn(fvol, dens);
        const double self = __dsub_rn(t1, __dmul_rn(t2, t2));
        U256 P;
#pragma unroll
        for (int k = 0; k < 4; ++k) P.w[k] = recw[(size_t)c * 4 + k];
        // P = sum_j W_ij |E_ij| / |c_j| * 2^171 ; penalty = that / (2W |c|)
        const double pen = __ddiv_rn(ldexp(u256_to_double(P), -128), __dmul_rn(W2, (double)size));
        acc.qds_self += fp_from_double(self, SC_QDS);
        acc.qds_pair += fp_from_double(pen, SC_QDS);
        acc.dens += fp_from_double(dens, SC_MEAN);
        acc.contr += fp_from_double(contr, SC_MEAN);
        acc.expn += fp_from_double(expn, SC_MEAN);
        acc.cond += fp_from_double(cond, SC_MEAN);
        acc.vol2 += (u128)vol * (u128)vol;
        acc.ein += (unsigned long long)ein;
        acc.eout += (unsigned long long)eout;
        acc.nonempty += 1;
        acc.slots += rc[REC_SLOTS];
        acc.cnt2 += rc[REC_CNT2];
        qw += fp_from_double(qwt, SC_QDS);
        if (pc.size) pc.size[c] = size;
        if (pc.ein) pc.ein[c] = ein;
        if (pc.eout) pc.eout[c] = eout;
        if (pc.dens) pc.dens[c] = dens;
        if (pc.contr) pc.contr[c] = contr;
        if (pc.expn) pc.expn[c] = expn;
        if (pc.cond) pc.cond[c] = cond;
        if (pc.qds) pc.qds[c] = __dsub_rn(self, pen);
    }
    flush_terms(acc, qw, g, o);
}

// ---------------------------------------------------------------- load time

// Weight check and total: every weight must be 0 or in [2^-20, 2^20) (NaN
// fails); the fixed-point sum over all arcs (2 W * 2^43) goes to three limbs.
__global__ void k_wcheck(const float *__restrict__ wt, long long n_arcs, int *status, unsigned long long *lim)
{
    u128 s = 0;
    bool bad = false;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n_arcs;
         e += (long long)gridDim.x * blockDim.x) {
        const float w = wt[e];
        if (!(w == 0.0f || (w >= 9.5367431640625e-07f && w < 1048576.0f))) {
            bad = true;
            continue;
        }
        s += w_fixed(w);
    }
    if (bad) atomicOr(status, 2);
    for (int d = 16; d > 0; d >>= 1) s += shfl_down_u128(s, d);
    if ((threadIdx.x & 31) == 0 && s) limbs_add(lim, (i128)s);
}

// Symmetric weights: arc (u, v) and arc (v, u) carry the same weight (rows
// sorted, as the full validation has checked).
__global__ void k_wsym(const long long *__restrict__ row_ptr, const int *__restrict__ col,
                       const float *__restrict__ wt, long long n, int *status)
{
    bool bad = false;
    for (long long u = (long long)blockIdx.x * blockDim.x + threadIdx.x; u < n;
         u += (long long)gridDim.x * blockDim.x) {
        for (long long k = row_ptr[u]; k < row_ptr[u + 1] && !bad; ++k) {
            const int v = col[k];
            long long lo = row_ptr[v], hi = row_ptr[v + 1];
            bool found = false;
            while (lo < hi) {
                const long long mid = (lo + hi) >> 1;
                const int w = col[mid];
                if (w == (int)u) {
                    found = wt[mid] == wt[k];
                    break;
                }
                if (w < (int)u) lo = mid + 1; else hi = mid;
            }
            if (!found) bad = true;
        }
    }
    if (bad) atomicOr(status, 4);
}

