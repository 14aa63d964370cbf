// qm_rows.cuh -- phase A of the two-phase scoring pipeline in stored node order
// (included by qm_kernels.cu).
//
// The packed runs only need each community's segment base, the exclusive
// prefix of the communities' volumes, so no counting sort of the nodes is made:
// k_hist_vol (or the pass that permutes the labels of a renumbered graph)
// counts members and arcs of every community, a scan turns the arcs into
// segment bases, and k_rows walks the graph's rows in order.  A warp takes 32
// consecutive nodes, whose arcs are one contiguous range of the CSR; the lanes
// gather the far-end labels and append those that differ to their community's
// run through one 64-bit cursor a community (cut arcs above, packed labels
// below), one atomic per warp step and community.
//
// Against the member-order pass (a counting sort of the nodes with their
// degrees, a scan of the n degrees, rows in community order) this reads and
// writes 20 bytes a node less and streams the adjacency whatever the labels.
// The walk waits on the chain column -> label (-> pair) and issues about 50
// instructions per 32 arcs.  Measured, phase A without the label permutation:
// 10^8 nodes renumbered, planted, 8.1 -> 5.2 ms (the walk 6.7 -> 4.85); 10^7
// renumbered, 20% moved, 1.26 -> 0.85 ms; 10^7 as given 1.61 -> 1.18 ms.
// Included inside namespace qm of qm_kernels.cu, after the helpers it uses.

// Members and arcs of every community in node order, with the label range
// check (bit 0 of *status).  With few ids the counts are taken in shared
// memory (two words an id) and added once per block.
__global__ void k_hist_vol(const int *__restrict__ labels, const long long *__restrict__ row_ptr, long long n, int K,
                           unsigned long long *cv, int *status, int use_smem)
{
    extern __shared__ unsigned shv[];  // [K] members, [K] arcs
    if (use_smem) {
        for (int i = threadIdx.x; i < 2 * K; i += blockDim.x) shv[i] = 0u;
        block_sync();
    }
    bool bad = false;
    const int lane = threadIdx.x & 31;
    const long long nw = (long long)gridDim.x * (blockDim.x >> 5);
    for (long long i0 = (((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * (32 * HIST_UNROLL); i0 < n;
         i0 += nw * (32 * HIST_UNROLL)) {
        int l[HIST_UNROLL];
        unsigned d[HIST_UNROLL];
#pragma unroll
        for (int q = 0; q < HIST_UNROLL; ++q) {
            const long long i = i0 + q * 32 + lane;
            l[q] = i < n ? __ldcs(&labels[i]) : 0;
            d[q] = i < n ? (unsigned)(__ldg(&row_ptr[i + 1]) - __ldg(&row_ptr[i])) : 0u;
        }
#pragma unroll
        for (int q = 0; q < HIST_UNROLL; ++q) {
            const bool in = i0 + q * 32 + lane < n, ok = in && (unsigned)l[q] < (unsigned)K;
            if (in && !ok) bad = true;
            if (use_smem) {
                if (ok) {
                    atomicAdd(&shv[l[q]], 1u);
                    atomicAdd(&shv[K + l[q]], d[q]);
                }
            } else {
                vol_add_warp(cv, l[q], d[q], ok);
            }
        }
    }
    if (bad) atomicOr(status, 1);
    if (use_smem) {
        block_sync();
        for (int i = threadIdx.x; i < K; i += blockDim.x)
            if (shv[i]) atomicAdd(&cv[i], ((unsigned long long)shv[i] << VOL_BITS) | shv[K + i]);
    }
}

// k_permute_hist with the communities' arcs: labels of a renumbered graph
// gathered into its order, out[j] = labels[inv[j]], counted on the way (SHARED:
// in shared memory, see VOL_SMEM_IDS).
template <bool SHARED>
__global__ void k_permute_vol(const int *__restrict__ labels, const int *__restrict__ inv,
                              const long long *__restrict__ row_ptr, long long n, int *__restrict__ out, int K,
                              unsigned long long *cv, int *status)
{
    extern __shared__ unsigned shp[];  // SHARED: [K] members, [K] arcs
    if (SHARED) vol_smem_zero(shp, K);
    bool bad = false;
    const int lane = threadIdx.x & 31;
    const long long nw = (long long)gridDim.x * (blockDim.x >> 5);
    for (long long j0 = (((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * (32 * HIST_UNROLL); j0 < n;
         j0 += nw * (32 * HIST_UNROLL)) {
        int l[HIST_UNROLL];
        unsigned d[HIST_UNROLL];
#pragma unroll
        for (int q = 0; q < HIST_UNROLL; ++q) {
            const long long j = j0 + q * 32 + lane;
            l[q] = j < n ? __ldcs(&inv[j]) : 0;
            d[q] = j < n ? (unsigned)(__ldg(&row_ptr[j + 1]) - __ldg(&row_ptr[j])) : 0u;
        }
#pragma unroll
        for (int q = 0; q < HIST_UNROLL; ++q) l[q] = __ldg(&labels[l[q]]);
#pragma unroll
        for (int q = 0; q < HIST_UNROLL; ++q) {
            const long long j = j0 + q * 32 + lane;
            const bool in = j < n, ok = in && (unsigned)l[q] < (unsigned)K;
            if (in) out[j] = l[q];
            if (in && !ok) bad = true;
            if (SHARED) vol_smem_add_warp(shp, K, l[q], d[q], ok);
            else vol_add_warp(cv, l[q], d[q], ok);
        }
    }
    if (bad) atomicOr(status, 1);
    if (SHARED) vol_smem_flush(shp, K, cv);
}

// ------------------------------------------------------------------ segment bases

constexpr int VSCAN_THREADS = 512;
constexpr int VSCAN_PER = 8;                          // words a thread
constexpr int VSCAN_TILE = VSCAN_THREADS * VSCAN_PER;

__device__ __forceinline__ unsigned vscan_load(const unsigned long long *cv, long long b, int K, unsigned long long (&w)[VSCAN_PER])
{
    unsigned sum = 0;
#pragma unroll
    for (int k = 0; k < VSCAN_PER; ++k) {
        w[k] = b + k < K ? cv[b + k] : 0ull;
        sum += (unsigned)(w[k] & VOL_MASK);
    }
    return sum;
}

// Arcs of every tile of communities.
__global__ void __launch_bounds__(VSCAN_THREADS) k_vscan_tiles(const unsigned long long *cv, int K, unsigned *tile_sum,
                                                               const int *status)
{
    __shared__ unsigned long long red[72];
    if (*status) return;
    unsigned long long w[VSCAN_PER];
    const unsigned s = vscan_load(cv, (long long)blockIdx.x * VSCAN_TILE + threadIdx.x * VSCAN_PER, K, w);
    const unsigned t = (unsigned)group_sum_u64(s, VSCAN_THREADS, red);
    if (threadIdx.x == 0) tile_sum[blockIdx.x] = t;
}

// Segment base (arcs of the communities before) and reciprocal of every
// community; each block first adds the sums of the tiles before its own.
__global__ void __launch_bounds__(VSCAN_THREADS) k_vscan_apply(const unsigned long long *cv, int K,
                                                               const unsigned *tile_sum, unsigned *base, Rcp *recip,
                                                               const int *status)
{
    __shared__ unsigned long long red[72];
    if (*status) return;
    unsigned before = 0;
    if (blockIdx.x) {
        for (int t = threadIdx.x; t < (int)blockIdx.x; t += VSCAN_THREADS) before += tile_sum[t];
        before = (unsigned)group_sum_u64(before, VSCAN_THREADS, red);
        block_sync();
    }
    unsigned long long w[VSCAN_PER];
    const long long b = (long long)blockIdx.x * VSCAN_TILE + threadIdx.x * VSCAN_PER;
    const unsigned sum = vscan_load(cv, b, K, w);
    unsigned excl;
    group_exclusive_scan(sum, excl, VSCAN_THREADS, red);
    unsigned run = before + excl;
#pragma unroll
    for (int k = 0; k < VSCAN_PER; ++k) {
        if (b + k >= K) break;
        base[b + k] = run;
        run += (unsigned)(w[k] & VOL_MASK);
    }
    // the divisions, one community a thread at a time so that few communities spread over all threads
    for (int k = 0; k < VSCAN_PER; ++k) {
        const long long c = (long long)blockIdx.x * VSCAN_TILE + k * VSCAN_THREADS + threadIdx.x;
        if (c >= K) break;
        const long long s = (long long)(cv[c] >> VOL_BITS);
        if (s > 0) recip[c] = rcp_of(s);
    }
}

// ------------------------------------------------------------------ the walk

constexpr int ROWS_THREADS = 256;
// Arcs a lane gathers at a time within one community's rows, and resident
// blocks per SM: the gathers from the block encoding hit L2 and wait on a chain
// of two loads, so they take few arcs and all warps; the others more arcs.
// k_rows at 10^8 nodes, planted (block encoding): 4 arcs and 8 blocks 4.87 ms,
// 4 and 6 5.11, 6 and 5 5.00, 8 and 5 5.30, 8 and 6 5.68; at 10^7 nodes, 20%
// moved (packed copy): 8 and 6 0.784 ms, 8 and 5 0.854, 8 and 4 0.997.
template <int LAB> constexpr int rows_unroll() { return LAB == LAB_BLOCKS ? 4 : 8; }
template <bool WT, int LAB> constexpr int rows_blocks() { return WT ? 4 : LAB == LAB_BLOCKS ? 8 : 6; }
constexpr int ROWS_MIX_UNROLL = 4;  // and where the rows of a chunk belong to many
constexpr int ROWS_MAX_RUNS = 4;    // stretches of one label a chunk may have to be walked one by one
constexpr int ROWS_OWN_CAP = 2048;  // arcs of a mixed chunk

struct RowsArgs {
    const long long *row_ptr;
    const int *col;
    const int *labels;                // stored order
    const unsigned long long *plab;   // packed copy or block encoding, as LAB says
    long long n;
    const unsigned *base;             // [K] segment bases
    unsigned long long *curs;         // [K] cut arcs << 32 | packed labels (zeroed)
    int *nbr;                         // packed labels
    const int *status;
    const int *bx_bad;                // with the block encoding tried: whether it did not fit
    Shard own;
    const float *wt;                  // weighted graphs
    float *nbrw;
    unsigned long long *wl;
    int K;
};

// Labels of U far-end nodes v (with CHECK some may be -1: none, and stay so),
// all in flight together.
template <int LAB, int U, bool CHECK>
__device__ __forceinline__ void far_labels(const RowsArgs &a, int (&v)[U], unsigned long long keep)
{
    if (LAB == LAB_BLOCKS) {
        const int *words = (const int *)a.plab;
        int l[U];
        bool exc = false;
#pragma unroll
        for (int k = 0; k < U; ++k) l[k] = ld_hint(&words[(unsigned)(CHECK ? max(v[k], 0) : v[k]) >> 4], keep);
#pragma unroll
        for (int k = 0; k < U; ++k) exc |= l[k] < 0;
        if (__any_sync(0xffffffffu, exc)) {  // blocks of several labels
            // (loads under a predicate, not a branch: lanes with and without one stay together)
            const unsigned long long *pairs = a.plab + blk_pairs_at(a.n) / 2;
            const int *slots = words + blk_slots_at(a.n);
            unsigned long long p[U];
            bool many = false;
#pragma unroll
            for (int k = 0; k < U; ++k) {
                p[k] = 0ull;
                asm volatile("{\n\t.reg .pred q;\n\tsetp.ge.u32 q, %1, %2;\n\t"
                             "@q ld.global.nc.L2::cache_hint.b64 %0, [%3], %4;\n\t}"
                             : "+l"(p[k])
                             : "r"((unsigned)l[k]), "r"(BLK_PAIR), "l"(pairs + ((unsigned)l[k] & BLK_INDEX)), "l"(keep));
                many |= (unsigned)l[k] >= BLK_SLOT && (unsigned)l[k] < BLK_PAIR;
            }
#pragma unroll
            for (int k = 0; k < U; ++k) {
                const unsigned lo = (unsigned)p[k], hi = (unsigned)(p[k] >> 32);
                const bool second = (hi >> (10 + (v[k] & 15))) & 1u;
                const unsigned t = (second ? __funnelshift_r(lo, hi, PACK_BITS) : lo) & 0x1FFFFFu;
                if ((unsigned)l[k] >= BLK_PAIR) l[k] = (int)t;
            }
            if (__any_sync(0xffffffffu, many)) {  // blocks of three or more
#pragma unroll
                for (int k = 0; k < U; ++k)
                    if (l[k] < 0) l[k] = ld_hint(&slots[(((unsigned)l[k] & BLK_INDEX) << 4) + ((unsigned)v[k] & 15u)], keep);
            }
        }
#pragma unroll
        for (int k = 0; k < U; ++k) v[k] = CHECK && v[k] < 0 ? -1 : l[k];
        return;
    }
#pragma unroll
    for (int k = 0; k < U; ++k)
        if (!CHECK || v[k] >= 0) v[k] = LAB == LAB_PACK3 ? ld_label3(a.plab, v[k], keep) : ld_hint(&a.labels[v[k]], keep);
}

// One step of U arcs a lane, from arc e0 on, of nodes of community c, whose
// segment starts at cbase (CHECK: only arcs below e_hi).  The lanes' labels to
// pack are placed by one warp scan and one atomic.
template <bool WT, int LAB, bool HI, int U, bool CHECK>
__device__ __forceinline__ void rows_step(const RowsArgs &a, const int *col, const float *wt, unsigned e0, unsigned e_hi,
                                          int c, unsigned cbase, unsigned long long keep, int lane, u128 &w_in,
                                          u128 &w_out)
{
    int lab[U];
    float wv[U];
#pragma unroll
    for (int k = 0; k < U; ++k) {
        const unsigned e = e0 + lane + 32u * k;
        lab[k] = !CHECK || e < e_hi ? __ldcs(&col[e]) : -1;
        if (WT) wv[k] = !CHECK || e < e_hi ? __ldcs(&wt[e]) : 0.0f;
    }
    far_labels<LAB, U, CHECK>(a, lab, keep);
    unsigned cnt = 0;  // cut arcs << 16 | labels to pack
#pragma unroll
    for (int k = 0; k < U; ++k) {
        if (WT && (!CHECK || lab[k] >= 0)) {
            const unsigned long long f = w_fixed(wv[k]);
            if (lab[k] == c) w_in += f; else w_out += f;
        }
        if ((!CHECK || lab[k] >= 0) && lab[k] != c) cnt += HI ? 1u << 16 : (1u << 16) + 1u;
        if (HI && lab[k] > c) cnt += 1u;
    }
    unsigned inc = cnt;
#pragma unroll
    for (int s = 1; s < 32; s <<= 1) {
        const unsigned t = __shfl_up_sync(0xffffffffu, inc, s);
        if (lane >= s) inc += t;
    }
    const unsigned tot = __shfl_sync(0xffffffffu, inc, 31);
    if (!tot) return;
    unsigned at = 0;
    if (lane == 0)
        at = cbase + (unsigned)atomicAdd(&a.curs[c], ((unsigned long long)(tot >> 16) << 32) | (tot & 0xFFFFu));
    at = __shfl_sync(0xffffffffu, at, 0) + ((inc - cnt) & 0xFFFFu);
#pragma unroll
    for (int k = 0; k < U; ++k)
        if (HI ? lab[k] > c : ((!CHECK || lab[k] >= 0) && lab[k] != c)) {
            __stcs(&a.nbr[at], lab[k]);
            if (WT) __stcs(&a.nbrw[at], wv[k]);
            ++at;
        }
}

// Arcs [e_lo, e_hi) (relative to col) of nodes of community c: full steps, then
// the rest in a step of the same or half the size.
template <bool WT, int LAB, bool HI>
__device__ __forceinline__ void rows_one(const RowsArgs &a, const int *col, const float *wt, unsigned e_lo, unsigned e_hi,
                                         int c, unsigned cbase, unsigned long long keep, int lane, u128 &w_in,
                                         u128 &w_out)
{
    constexpr int U = rows_unroll<LAB>();
    unsigned e0 = e_lo;
    for (; e0 + 32u * U <= e_hi; e0 += 32u * U)
        rows_step<WT, LAB, HI, U, false>(a, col, wt, e0, e_hi, c, cbase, keep, lane, w_in, w_out);
    if (e_hi - e0 > 16u * U)
        rows_step<WT, LAB, HI, U, true>(a, col, wt, e0, e_hi, c, cbase, keep, lane, w_in, w_out);
    else if (e0 < e_hi)
        rows_step<WT, LAB, HI, U / 2, true>(a, col, wt, e0, e_hi, c, cbase, keep, lane, w_in, w_out);
}

// The arcs [0, total) of a chunk whose nodes belong to many communities: each
// arc's node is tabulated (own), and the lanes of one community take their
// places with one atomic.  On a weighted graph an arc's table entry is marked
// when it is cut, for rows_mixed_weights.
constexpr unsigned char ROWS_CUT = 0x80;

template <bool WT, int LAB, bool HI>
__device__ __forceinline__ void rows_mixed(const RowsArgs &a, const int *col, const float *wt, unsigned total,
                                           unsigned char *own, const int *cw, const unsigned *bw,
                                           unsigned long long keep, int lane)
{
    const unsigned lt = (1u << lane) - 1u;
    for (unsigned e0 = 0; e0 < total; e0 += 32u * ROWS_MIX_UNROLL) {
        int lab[ROWS_MIX_UNROLL], o[ROWS_MIX_UNROLL];
        float wv[ROWS_MIX_UNROLL];
        unsigned peers[ROWS_MIX_UNROLL], hm[ROWS_MIX_UNROLL], at[ROWS_MIX_UNROLL];
#pragma unroll
        for (int k = 0; k < ROWS_MIX_UNROLL; ++k) {
            const unsigned e = e0 + lane + 32u * k;
            lab[k] = e < total ? __ldcs(&col[e]) : -1;
            if (WT) wv[k] = e < total ? __ldg(&wt[e]) : 0.0f;
            o[k] = e < total ? own[e] : 0;
        }
        far_labels<LAB, ROWS_MIX_UNROLL, true>(a, lab, keep);
#pragma unroll
        for (int k = 0; k < ROWS_MIX_UNROLL; ++k) {
            const int c = cw[o[k]];
            const bool out = lab[k] >= 0 && lab[k] != c;
            if (WT && out) own[e0 + lane + 32u * k] |= ROWS_CUT;
            const bool cut = out && a.own.owns(c), pack = cut && (!HI || lab[k] > c);
            const unsigned cm = __ballot_sync(0xffffffffu, cut);
            hm[k] = __ballot_sync(0xffffffffu, pack);
            peers[k] = __match_any_sync(0xffffffffu, c) & cm;
            if (!cut) peers[k] = 0u;
            at[k] = 0u;
            if (cut && lane == __ffs(peers[k]) - 1)
                at[k] = bw[o[k]] + (unsigned)atomicAdd(&a.curs[c], ((unsigned long long)__popc(peers[k]) << 32) |
                                                                        (unsigned)__popc(peers[k] & hm[k]));
        }
#pragma unroll
        for (int k = 0; k < ROWS_MIX_UNROLL; ++k) {
            const unsigned b = __shfl_sync(0xffffffffu, at[k], peers[k] ? __ffs(peers[k]) - 1 : 0);
            if (peers[k] && ((hm[k] >> lane) & 1u)) {
                const unsigned q = b + __popc(peers[k] & hm[k] & lt);
                __stcs(&a.nbr[q], lab[k]);
                if (WT) __stcs(&a.nbrw[q], wv[k]);
            }
        }
    }
}

// Intra and cut weight sums of a mixed chunk, a lane per node over its arcs
// [rel, end) (the chunk's weights are in L1 by then), added to its community's
// sums.
__device__ __forceinline__ void rows_mixed_weights(const RowsArgs &a, const WeightSums &ws, const float *wt,
                                                   const unsigned char *own, unsigned rel, unsigned end, int c, bool node)
{
    if (!node || rel == end || !a.own.owns(c)) return;
    u128 w_in = 0, w_out = 0;
    for (unsigned e = rel; e < end; ++e) {
        const unsigned long long f = w_fixed(__ldg(&wt[e]));
        if (own[e] & ROWS_CUT) w_out += f; else w_in += f;
    }
    ws.add(c, w_in, w_out);
}

// Up to this many label ids a block adds up their weights in shared memory: a
// node of a mixed chunk (a stretch, where rows are long) adds up to six words,
// and with few communities all SMs' additions queue for few of them.  The call at
// 2*10^6 nodes as given, two communities in turn, global words against shared: 2.59
// and 0.37 ms; ten 1.60 and 0.37, a hundred 0.52 and 0.37 (a thousand, global: 0.38).
constexpr int ROWS_W_IDS = 256;

template <bool WT, int LAB, bool HI>
__global__ void __launch_bounds__(ROWS_THREADS, (rows_blocks<WT, LAB>())) k_rows(RowsArgs a)
{
    __shared__ int cw_s[ROWS_THREADS / 32][32];
    __shared__ unsigned bw_s[ROWS_THREADS / 32][32];
    __shared__ unsigned char own_s[ROWS_THREADS / 32][ROWS_OWN_CAP];
    __shared__ unsigned wsum_s[WT ? ROWS_W_IDS * 6 : 1];
    if (*a.status) return;
    if (a.bx_bad && (LAB == LAB_BLOCKS) == (*a.bx_bad != 0)) return;
    const WeightSums ws{a.wl, WT && a.K <= ROWS_W_IDS ? wsum_s : nullptr};
    if (WT && ws.smem) {
        for (int i = threadIdx.x; i < a.K * 6; i += ROWS_THREADS) wsum_s[i] = 0u;
        block_sync();
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned long long keep = l2_policy_evict_last();
    const long long nwarps = (long long)gridDim.x * (ROWS_THREADS / 32);
    for (long long u0 = ((long long)blockIdx.x * (ROWS_THREADS / 32) + w) * 32; u0 < a.n; u0 += nwarps * 32) {
        const int nm = (int)min(32LL, a.n - u0);
        const long long u = u0 + min(lane, nm - 1);
        const long long r = __ldg(&a.row_ptr[u]), r0 = __shfl_sync(0xffffffffu, r, 0);
        const unsigned total = (unsigned)(__ldg(&a.row_ptr[u0 + nm]) - r0);
        const unsigned rel = lane < nm ? (unsigned)(r - r0) : total;
        const int c = ld_hint(&a.labels[u], keep);
        const int prev = __shfl_up_sync(0xffffffffu, c, 1);
        const unsigned heads = __ballot_sync(0xffffffffu, lane < nm && (lane == 0 || c != prev));
        if (total == 0u) continue;
        const unsigned bs = __ldg(&a.base[c]);
        const int *col = a.col + r0;
        if (__popc(heads) <= ROWS_MAX_RUNS || total > (unsigned)ROWS_OWN_CAP) {
            unsigned rem = heads;
            while (rem) {
                const int lo = __ffs(rem) - 1;
                rem &= rem - 1;
                const int hi = rem ? __ffs(rem) - 1 : nm;
                const unsigned e_lo = __shfl_sync(0xffffffffu, rel, lo);
                const unsigned e_hi = hi < 32 ? __shfl_sync(0xffffffffu, rel, hi) : total;
                const int cc = __shfl_sync(0xffffffffu, c, lo);
                const unsigned cb = __shfl_sync(0xffffffffu, bs, lo);
                if (e_lo == e_hi || !a.own.owns(cc)) continue;
                u128 w_in = 0, w_out = 0;
                rows_one<WT, LAB, HI>(a, col, WT ? a.wt + r0 : nullptr, e_lo, e_hi, cc, cb, keep, lane, w_in, w_out);
                if (WT) flush_weights(ws, cc, w_in, w_out, lane);
            }
        } else {
            __syncwarp();
            cw_s[w][lane] = c;
            bw_s[w][lane] = bs;
            const unsigned nxt = __shfl_down_sync(0xffffffffu, rel, 1);
            const unsigned end = lane == 31 ? total : nxt;
            if (lane < nm)
                for (unsigned e = rel; e < end; ++e) own_s[w][e] = (unsigned char)lane;
            __syncwarp();
            rows_mixed<WT, LAB, HI>(a, col, WT ? a.wt + r0 : nullptr, total, own_s[w], cw_s[w], bw_s[w], keep, lane);
            __syncwarp();
            if (WT) {
                rows_mixed_weights(a, ws, a.wt + r0, own_s[w], rel, end, c, lane < nm);
                __syncwarp();
            }
        }
    }
    if (WT && ws.smem) {
        block_sync();
        for (int i = threadIdx.x; i < a.K * 2; i += ROWS_THREADS) {  // intra and cut sums
            const unsigned *L = wsum_s + 3 * i;
            wsum_add(a.wl + 3 * (size_t)i, ((u128)L[2] << 64) | ((u128)L[1] << 32) | (u128)L[0]);
        }
    }
}

// One header per non-empty owned community, by run length (as k_classify), from
// the volumes and cursors of the walk; the cut arcs go to inter[] for the
// records.
__global__ void k_rows_classify(const unsigned long long *cv, const unsigned *base, const unsigned long long *curs,
                                const int *half_len, int K,
                                int warp_fill, int group_fill, int block_fill, RunHdr *big, RunHdr *small, RunHdr *lng,
                                RunHdr *mid, int *inter, int *counters, const int *status, Shard own)
{
    if (*status) return;
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    for (long long c0 = (long long)blockIdx.x * blockDim.x; c0 < K; c0 += (long long)gridDim.x * blockDim.x) {
        const long long cl = c0 + threadIdx.x;
        int cls = -1;
        RunHdr h{-1, 0u, 0u, 0u};
        if (cl < K) {
            const int c = (int)cl;
            const unsigned long long v = cv[c];
            if ((v >> VOL_BITS) != 0ull && own.owns(c)) {
                const unsigned vol = (unsigned)(v & VOL_MASK);
                if (half_len) {  // half-edge gathers left 2|E_c^in|: the cut arcs are the rest of the volume
                    h = RunHdr{c, base[c], (unsigned)half_len[c], vol};
                    inter[c] = (int)(vol - (unsigned)inter[c]);
                } else {
                    const unsigned long long q = curs[c];
                    h = RunHdr{c, base[c], (unsigned)q, vol};
                    inter[c] = (int)(q >> 32);
                }
                cls = h.m > (unsigned)block_fill ? 2
                      : h.m > (unsigned)group_fill ? 0
                      : h.m > (unsigned)warp_fill ? 3 : 1;
            }
        }
        const int ctr[4] = {C_BIG_COUNT, C_SMALL_COUNT, C_LONG_COUNT, C_MID_COUNT};
        RunHdr *const lists[4] = {big, small, lng, mid};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const unsigned mask = __ballot_sync(0xffffffffu, cls == k);
            if (!mask) continue;
            const int leader = __ffs(mask) - 1;
            int b = 0;
            if (lane == leader) b = atomicAdd(&counters[ctr[k]], __popc(mask));
            b = __shfl_sync(0xffffffffu, b, leader);
            if (cls == k) lists[k][b + __popc(mask & lt)] = h;
        }
    }
}
