// qm_cover.cu -- the metrics of a cover (overlapping communities).
//
// The paper leaves overlapping communities to future work (Sec. VI); its
// formulas are written with node sets, and a cover is scored by reading them
// literally: |c| its members, |E_c^in| the edges with both ends in c,
// |E_c^out| those with exactly one end in c, |E_ci,cj| those that leave c_i
// and enter c_j (u in c_i \ c_j, v in c_j \ c_i), |c n c'| the nodes in both,
// and a pair of nodes "in the same community" when the two share one.
//
// Scoring (Eqs. 8-9, Sec. II-B.3): the cover is brought to the graph's stored
// order and scored by the partition path's two phases.  k_cover_walk takes the
// rows in node order; for every arc and every community c of its near end it
// tests the far end's list for c, counts the arc as cut, and packs into c's run
// the communities j > c of the far end that the near end is not in (each
// unordered pair is charged to its smaller id).  A run's segment is sized by
// the list lengths of its members' neighbours (k_cover_cap).  The counting,
// the terms and the sums are the partition path's, so a cover with one
// community per node gives the partition's bits.  Covers with long lists, ones
// whose segments do not fit the scratch, and ones of 2^20 ids or more, are transposed
// into member lists and scored by one block per community (k_cover_score).
// Measured, 10^6 nodes, a tenth of them in two communities: 2.46 ms by member
// lists, 0.60 by runs (k_cover_walk 0.27, k_cover_cap 0.14, counting 0.07); the
// walk is bound by the instructions of its rounds (two for most warps), the
// segment sizes by their atomics.
//
// Comparison (Eqs. 1-7): one block per truth community counts the cells
// |a n b| over its members' found lists; rows and columns add the entropy, F
// and NVD terms.  The pair counts come from the cells and sizes as for a
// partition (sum C(|a n b|, 2) counts a pair once per cell holding both), less
// a correction over pairs of nodes that share two or more communities on one
// side: such pairs can only be formed by nodes with two or more memberships,
// which each block lists and pairs up.
#include <algorithm>
#include <climits>

#include "qm_batched.h"
#include "qm_cover.h"
#include "qm_community.cuh"
#include "qm_finalize.cuh"

namespace qm {
using namespace qmk;

namespace {

constexpr int COVER_THREADS = 256;
constexpr int COVER_SMEM = 48 * 1024;
// Covers with a longer list than this are scored by member lists: k_cover_walk
// turns the two ends' lists in step over the 32 arcs of a warp, so that one arc's
// pairs of communities are walked by all.  5*10^5 nodes, every 500th in L
// communities, by runs and by member lists, ms: L = 8 0.46 and 1.50, 16 0.74 and
// 1.59, 32 2.53 and 1.78, 128 88 and 4.6.
constexpr int COVER_LIST_MAX = 16;
// Memberships of both covers from which a comparison tabulates log(N / n) and n / N.
constexpr long long COVER_TABLE_MEMB = 1 << 15;
constexpr int OVL_CAP = 2048;  // overlapping members of one community paired in shared memory

// extra accumulator words after the GC_* words of a comparison
enum { GC_SAME_A_CORR = GC_COUNT, GC_SAME_B_CORR = GC_COUNT + 1, GC_A11_CORR = GC_COUNT + 2, GC_WORDS = GC_COUNT + 3 };
enum { CC_NEXT_A = 0, CC_NEXT_B = 1, CC_NEXT_C = 2, CC_GATE = 3, CC_OLD = 4, CC_LONG = 5, CC_TOTAL = 6 /* two words */,
       CC_SCAN = 8, CC_RUNS = 16, CC_HUBS = 32 };

size_t al(size_t x) { return (x + 255) / 256 * 256; }

void carve_side(char *&p, CoverSide &c, long long n, long long m, int K)
{
    c.off = (int *)p;
    p += al(((size_t)n + 1) * 4);
    c.memb = (int *)p;
    p += al((size_t)std::max(m, 1LL) * 4);
    c.len = (int *)p;
    p += al(((size_t)n + 1) * 4);
    c.cstart = (int *)p;
    p += al(((size_t)K + 1) * 4);
    c.cmem = (int *)p;
    p += al((size_t)std::max(m, 1LL) * 4);
    c.K = K;
}

}  // namespace

// Entries of the packed runs' scratch: what covers whose memberships do not
// follow the degrees need (every arc once per pair of its ends' communities),
// and a quarter more.
// Small calls keep the member lists: the runs take nine launches more, and pay from
// about 2^20 arcs on, or where a community's arcs are many for its one block (us a
// call, lists and runs: 20,000 nodes 0.38*10^6 arcs 197-231 and 243-262, 40,000
// nodes 244-275 and 248-271, 10^5 nodes 270-345 and 272-288; few communities, 5,000
// nodes, 19,000 arcs each 379-931 and 218-372, 9,500 each 379-458 and 208-231).
long long cover_run_entries(long long n, long long n_arcs, long long m, int K)
{
    if (!cover_runs_ok(K) || (n_arcs < (1LL << 20) && n_arcs < (1LL << 12) * K)) return 0;
    const double r = std::max(1.0, (double)m / (double)n);
    const double e = 1.25 * (double)n_arcs * r * r + 4096.0;
    return e < 4.0e9 ? (long long)e : 0;
}

size_t cover_score_ws_bytes(long long n, long long m, int K, long long run_entries)
{
    return carve_cover_score_ws(reinterpret_cast<void *>(4096), n, m, K, run_entries).bytes;
}

CoverWs carve_cover_score_ws(void *base, long long n, long long m, int K, long long run_entries)
{
    CoverWs w{};
    char *p = (char *)base;
    w.status = (int *)p;
    w.counters = (int *)(p + 16);
    p += 256;
    w.gacc = (unsigned long long *)p;
    p += al(64 * 8);
    w.result = p;
    p += al(sizeof(qm_quality));
    w.a.size = (int *)p;
    p += al((size_t)K * 4);
    w.a.cur = (int *)p;
    p += al((size_t)K * 4);
    if (run_entries) {
        w.cv = (unsigned long long *)p;
        p += al((size_t)K * 8);
        w.capw = (unsigned long long *)p;
        p += al((size_t)K * 8);
        w.curs = (unsigned long long *)p;
        p += al((size_t)K * 8);
    }
    w.zero_bytes = (size_t)(p - (char *)base);
    carve_side(p, w.a, n, m, K);
    w.recip = (Rcp *)p;
    p += al((size_t)K * 16);
    w.run_entries = run_entries;
    if (run_entries) {
        w.head = (int *)p;
        p += al((size_t)n * 4);
        w.hubs = (int *)p;
        p += al((size_t)(run_entries / COVER_HUB + 1) * 4);  // (run_entries exceeds the arcs)
        w.base = (unsigned *)p;
        p += al((size_t)K * 4);
        w.inter = (int *)p;
        p += al((size_t)K * 4);
        w.rec = (unsigned long long *)p;
        p += al((size_t)K * REC_WORDS * 8);
        for (int k = 0; k < 4; ++k) {
            w.hdr[k] = (RunHdr *)p;
            p += al((size_t)K * sizeof(RunHdr));
        }
        w.nbr = (int *)p;
        p += al((size_t)run_entries * 4) + 256;
    }
    w.scan_tmp = (int *)p;
    p += al((scan_tmp_elems(std::max<long long>(n + 1, K)) + 64) * 4);
    w.bytes = (size_t)(p - (char *)base);
    return w;
}

size_t cover_compare_ws_bytes(long long n, long long ma, int ka, long long mb, int kb)
{
    return carve_cover_compare_ws(reinterpret_cast<void *>(4096), n, ma, ka, mb, kb).bytes;
}

CoverWs carve_cover_compare_ws(void *base, long long n, long long ma, int ka, long long mb, int kb)
{
    CoverWs w{};
    char *p = (char *)base;
    w.status = (int *)p;
    w.counters = (int *)(p + 16);
    p += 256;
    w.gacc = (unsigned long long *)p;
    p += al(64 * 8);
    w.result = p;
    p += al(sizeof(qm_compare));
    w.a.size = (int *)p;
    p += al((size_t)ka * 4);
    w.a.cur = (int *)p;
    p += al((size_t)ka * 4);
    w.b.size = (int *)p;
    p += al((size_t)kb * 4);
    w.b.cur = (int *)p;
    p += al((size_t)kb * 4);
    w.colmax = (unsigned *)p;
    p += al((size_t)kb * 4);
    w.zero_bytes = (size_t)(p - (char *)base);
    carve_side(p, w.a, n, ma, ka);
    carve_side(p, w.b, n, mb, kb);
    w.rowmax = (unsigned *)p;
    p += al((size_t)ka * 4);
    w.rowbest = (unsigned long long *)p;
    p += al((size_t)ka * 8);
    w.logt = (double *)p;
    p += al((size_t)LOGT_WORDS * 8);
    w.scan_tmp = (int *)p;
    p += al((scan_tmp_elems(std::max<long long>(n + 1, std::max(ka, kb))) + 64) * 4);
    w.bytes = (size_t)(p - (char *)base);
    return w;
}

// ------------------------------------------------------------------ bringing a cover to the stored order

// List length of every stored node (its caller node's list when the graph is
// renumbered), with the offsets' checks (non-decreasing from 0 to m).  *too_long
// (when wanted) is set where a list is longer than COVER_LIST_MAX.
__global__ void k_cover_len(const long long *mptr, long long n, long long m, const int *inv, int *len, int *status,
                            int *too_long)
{
    const long long stride = (long long)gridDim.x * blockDim.x;
    bool bad = false, above = false;
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += stride) {
        const long long u = inv ? (long long)__ldg(&inv[j]) : j;
        const long long b = __ldg(&mptr[u]), e = __ldg(&mptr[u + 1]);
        if (b < 0 || e < b || e > m || e - b > INT_MAX) {
            bad = true;
            len[j] = 0;
        } else {
            len[j] = (int)(e - b);
            above |= e - b > COVER_LIST_MAX;
        }
        if (j == 0 && (__ldg(&mptr[0]) != 0 || __ldg(&mptr[n]) != m)) bad = true;
    }
    if (bad) atomicOr(status, 1);
    if (too_long && above) *too_long = 1;
}

// Copies every stored node's list to its new offset, checks it (ids in [0, K),
// strictly increasing) and counts the community sizes.
// head[j] (when wanted): the id of a list of one, -1 for an empty list, else the
// list's offset with the sign bit set; and the nodes of more than COVER_HUB arcs
// are listed in hubs.
__global__ void k_cover_copy(const long long *mptr, const int *memb, long long n, const int *inv, int K,
                             const int *off, int *out, int *size, int *status, int *head,
                             const long long *__restrict__ row_ptr, int *hubs, int *nhubs)
{
    if (*(volatile int *)status) return;
    const long long stride = (long long)gridDim.x * blockDim.x;
    bool bad = false;
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += stride) {
        const long long u = inv ? (long long)__ldg(&inv[j]) : j;
        const long long b = __ldg(&mptr[u]);
        const int o = __ldg(&off[j]), len = __ldg(&off[j + 1]) - o;
        int prev = -1;
        for (int k = 0; k < len; ++k) {
            const int c = __ldg(&memb[b + k]);
            if (c < 0 || c >= K || c <= prev) {
                bad = true;
                break;
            }
            prev = c;
            out[o + k] = c;
            atomicAdd(&size[c], 1);
        }
        if (head) {
            head[j] = len == 1 ? prev : len == 0 ? -1 : (int)(0x80000000u | (unsigned)o);
            if (__ldg(&row_ptr[j + 1]) - __ldg(&row_ptr[j]) > COVER_HUB) hubs[atomicAdd(nhubs, 1)] = (int)j;
        }
    }
    if (bad) atomicOr(status, 1);
}

// Members of every community: node j into its communities' lists.
// (run_if: only when that flag is set.)
__global__ void k_cover_scatter(const int *off, const int *memb, long long n, const int *cstart, int *cur, int *cmem,
                                const int *status, const int *run_if)
{
    if (*status || (run_if && !*run_if)) return;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += stride)
        for (int k = __ldg(&off[j]); k < __ldg(&off[j + 1]); ++k) {
            const int c = __ldg(&memb[k]);
            cmem[__ldg(&cstart[c]) + atomicAdd(&cur[c], 1)] = (int)j;
        }
}

__global__ void k_cover_rcp(const int *size, int K, Rcp *recip, const int *status, const int *run_if)
{
    if (*status || (run_if && !*run_if)) return;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < K; c += gridDim.x * blockDim.x)
        recip[c] = size[c] > 0 ? rcp_of(size[c]) : Rcp{0ull, 0ull};
}

// ------------------------------------------------------------------ device helpers

__device__ __forceinline__ bool list_has(const int *l, int len, int c)
{
    for (int k = 0; k < len; ++k) {
        const int x = __ldg(&l[k]);
        if (x == c) return true;
        if (x > c) return false;
    }
    return false;
}

// |x n y| of two sorted lists, and their smallest common id (INT_MAX if none).
__device__ __forceinline__ int list_meet(const int *x, int lx, const int *y, int ly, int *first)
{
    int i = 0, j = 0, k = 0;
    *first = INT_MAX;
    while (i < lx && j < ly) {
        const int a = __ldg(&x[i]), b = __ldg(&y[j]);
        if (a == b) {
            if (k == 0) *first = a;
            ++k;
            ++i;
            ++j;
        } else if (a < b) {
            ++i;
        } else {
            ++j;
        }
    }
    return k;
}

// The block's next community from a shared claim counter (every thread gets it).
__device__ __forceinline__ int claim_next(int *counter, int *slot)
{
    block_sync();
    if (threadIdx.x == 0) *slot = atomicAdd(counter, 1);
    block_sync();
    return *slot;
}

// ------------------------------------------------------------------ scoring in node order

// Length of node v's list from its head word.
__device__ __forceinline__ int head_len(int h, const int *off, int v)
{
    if (h >= 0) return 1;
    return h == -1 ? 0 : __ldg(&off[v + 1]) - (h & 0x7FFFFFFF);
}

// Pieces of the rows of hubs (see COVER_HUB), which all warps take in turn.
constexpr unsigned HUB_PIECE = 2048;

// Members and arcs (cv) of every community, and members and segment size
// (capw): for each of its members the list lengths of the neighbours, summed.
// A warp takes 32 nodes, a lane per arc of one node at a time, then the hubs'
// rows in pieces.  The segments' total goes to *total.
__global__ void __launch_bounds__(256) k_cover_cap(const long long *__restrict__ row_ptr, const int *__restrict__ col,
                                                   const int *__restrict__ off, const int *__restrict__ memb,
                                                   const int *__restrict__ head, long long n, unsigned long long *cv,
                                                   unsigned long long *capw, unsigned long long *total,
                                                   const int *__restrict__ hubs, const int *nhubs,
                                                   const int *too_long, const int *status)
{
    if (*status || *too_long) return;
    const int lane = threadIdx.x & 31;
    const long long nw = (long long)gridDim.x * (blockDim.x >> 5);
    unsigned long long sum = 0;
    for (long long u0 = (((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32; u0 < n; u0 += nw * 32) {
        const long long u = min(u0 + lane, n - 1);
        const long long r = __ldg(&row_ptr[u]);
        const unsigned deg = (unsigned)(__ldg(&row_ptr[u + 1]) - r);
        unsigned long long mine = 0;
        const int cnt = (int)min(32LL, n - u0);
        for (int i0 = 0; i0 < cnt; i0 += 4) {
            unsigned s[4] = {0u, 0u, 0u, 0u};
            bool more = false;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const long long ri = __shfl_sync(0xffffffffu, r, i0 + q);
                unsigned d = i0 + q < cnt ? __shfl_sync(0xffffffffu, deg, i0 + q) : 0u;
                if (d > (unsigned)COVER_HUB) d = 0u;
                if ((unsigned)lane < d) {
                    const int v = __ldg(&col[ri + lane]);
                    s[q] = (unsigned)head_len(__ldg(&head[v]), off, v);
                }
                more |= d > 32u;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const unsigned t = __reduce_add_sync(0xffffffffu, s[q]);
                if (lane == i0 + q) mine = t;
            }
            if (more)  // rows of more than 32 arcs: the rest
                for (int q = 0; q < 4 && i0 + q < cnt; ++q) {
                    const long long ri = __shfl_sync(0xffffffffu, r, i0 + q);
                    const unsigned d = __shfl_sync(0xffffffffu, deg, i0 + q);
                    for (unsigned e0 = 32u; e0 < d && d <= (unsigned)COVER_HUB; e0 += 32u) {
                        unsigned x = 0u;
                        if (e0 + lane < d) {
                            const int v = __ldg(&col[ri + e0 + lane]);
                            x = (unsigned)head_len(__ldg(&head[v]), off, v);
                        }
                        const unsigned t = __reduce_add_sync(0xffffffffu, x);
                        if (lane == i0 + q) mine += t;
                    }
                }
        }
        if (lane < cnt) {
            const int b = __ldg(&off[u]), e = __ldg(&off[u + 1]);
            for (int k = b; k < e; ++k) {
                const int c = __ldg(&memb[k]);
                atomicAdd(&cv[c], (1ull << VOL_BITS) | deg);
                atomicAdd(&capw[c], (1ull << VOL_BITS) | mine);  // (a sum beyond 33 bits is beyond the scratch too)
            }
            sum += mine * (unsigned long long)(e - b);
        }
    }
    const long long wg = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    for (int i = 0; i < *nhubs; ++i) {
        const int u = __ldg(&hubs[i]), b = __ldg(&off[u]), len = __ldg(&off[u + 1]) - b;
        const long long r = __ldg(&row_ptr[u]), end = __ldg(&row_ptr[u + 1]);
        for (long long e0 = r + (wg + i) % nw * HUB_PIECE; e0 < end; e0 += nw * HUB_PIECE) {
            unsigned x = 0u;
#pragma unroll 4
            for (unsigned e = lane; e < HUB_PIECE; e += 32u) {
                const int v = e0 + e < end ? __ldg(&col[e0 + e]) : -1;
                if (v >= 0) x += (unsigned)head_len(__ldg(&head[v]), off, v);
            }
            const unsigned long long t = __reduce_add_sync(0xffffffffu, x);
            for (int k = lane; k < len; k += 32) atomicAdd(&capw[__ldg(&memb[b + k])], t);
            if (lane == 0) sum += t * (unsigned long long)len;
        }
    }
    sum = warp_sum_u64(sum);
    if (lane == 0 && sum) atomicAdd(total, sum);
}

// gate: nonzero keeps the kernels over runs from working; old_path: set when
// the cover is to be scored by member lists instead.
__global__ void k_cover_gate(const int *status, const unsigned long long *total, long long entries, const int *too_long,
                             int *gate, int *old_path)
{
    const bool fits = entries > 0 && *total <= (unsigned long long)entries && !*too_long;
    *gate = *status | (fits ? 0 : 256);
    *old_path = *status || fits ? 0 : 1;
}

struct CoverWalkArgs {
    const long long *row_ptr;
    const int *col, *off, *memb, *head;
    long long n;
    const unsigned *base;
    unsigned long long *curs;  // cut arcs << 32 | packed entries of each community
    int *nbr;
    const int *hubs, *nhubs;
    const int *gate;
};

constexpr int CW_THREADS = 256;
constexpr int CW_UNROLL = 4;
constexpr int CW_OWN_CAP = 2048;

// The arcs col[0 .. total) of a warp's nodes, node_of(e) the owner of arc e
// (0 .. 31), aoff the owners' list offsets (33).  Every arc is taken once per
// community c of its owner; each such visit adds one to c's cut arcs unless the
// far end is in c, and packs the far end's communities above c that the owner
// is not in.  The loops over the lists are warp-uniform (one turn each where
// all lists hold one id); the lanes of one community take their places with
// one atomic.
template <class OWN>
__device__ __forceinline__ void cover_arcs(const CoverWalkArgs &a, const int *col, unsigned total, const int *aoff,
                                           OWN node_of, int lane)
{
    constexpr unsigned ALL = 0xffffffffu;
    const unsigned lt = (1u << lane) - 1u;
    for (unsigned e0 = 0; e0 < total; e0 += 32u * CW_UNROLL) {
        int v[CW_UNROLL], hv[CW_UNROLL], o[CW_UNROLL];
#pragma unroll
        for (int k = 0; k < CW_UNROLL; ++k) {
            const unsigned e = e0 + lane + 32u * k;
            v[k] = e < total ? __ldcs(&col[e]) : -1;
            o[k] = e < total ? node_of(e) : 0;
        }
#pragma unroll
        for (int k = 0; k < CW_UNROLL; ++k) hv[k] = v[k] >= 0 ? __ldg(&a.head[v[k]]) : -1;
#pragma unroll
        for (int k = 0; k < CW_UNROLL; ++k) {
            const int ab = aoff[o[k]], la = v[k] >= 0 ? aoff[o[k] + 1] - ab : 0;
            const int h = hv[k], lb = v[k] >= 0 ? head_len(h, a.off, v[k]) : 0;
            const int *A = a.memb + ab, *B = a.memb + (h & 0x7FFFFFFF);
            const unsigned xa = __reduce_max_sync(ALL, (unsigned)la), yb = max(1u, __reduce_max_sync(ALL, (unsigned)lb));
            for (unsigned x = 0; x < xa; ++x) {
                const int c = (int)x < la ? __ldg(&A[x]) : -1;
                bool cut = c >= 0 && (lb == 1 ? h != c : !list_has(B, lb, c));
                __syncwarp();
                for (unsigned y = 0; y < yb; ++y) {
                    int j = -1;
                    if (cut && (int)y < lb) j = lb == 1 ? h : __ldg(&B[y]);
                    bool pack = j > c;
                    if (pack && la > 1) pack = !list_has(A, la, j);
                    __syncwarp();
                    const unsigned pm = __ballot_sync(ALL, pack), cm = y == 0 ? __ballot_sync(ALL, cut) : 0u;
                    if (!(pm | cm)) continue;
                    const unsigned same = __match_any_sync(ALL, c);
                    const unsigned peers = same & (pm | cm);
                    unsigned at = 0;
                    if ((peers >> lane) & 1u) {
                        if (lane == __ffs(peers) - 1)
                            at = __ldg(&a.base[c]) +
                                 (unsigned)atomicAdd(&a.curs[c], ((unsigned long long)__popc(same & cm) << 32) |
                                                                      (unsigned)__popc(same & pm));
                    }
                    at = __shfl_sync(ALL, at, peers ? __ffs(peers) - 1 : 0);
                    if (pack) __stcs(&a.nbr[at + __popc(same & pm & lt)], j);
                }
            }
        }
    }
}

__global__ void __launch_bounds__(CW_THREADS) k_cover_walk(CoverWalkArgs a)
{
    __shared__ int aoff_s[CW_THREADS / 32][33];
    __shared__ unsigned char own_s[CW_THREADS / 32][CW_OWN_CAP];
    if (*a.gate) return;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long long nwarps = (long long)gridDim.x * (CW_THREADS / 32);
    for (long long u0 = ((long long)blockIdx.x * (CW_THREADS / 32) + w) * 32; u0 < a.n; u0 += nwarps * 32) {
        const int nm = (int)min(32LL, a.n - u0);
        const long long u = u0 + min(lane, nm - 1);
        const long long r = __ldg(&a.row_ptr[u]), r0 = __shfl_sync(0xffffffffu, r, 0);
        const unsigned total = (unsigned)(__ldg(&a.row_ptr[u0 + nm]) - r0);
        const unsigned rel = lane < nm ? (unsigned)(r - r0) : total;
        const unsigned nxt = __shfl_down_sync(0xffffffffu, rel, 1), end = lane == 31 ? total : nxt;
        aoff_s[w][lane] = __ldg(&a.off[u0 + min(lane, nm)]);
        if (lane == 0) aoff_s[w][32] = __ldg(&a.off[u0 + nm]);
        __syncwarp();
        if (total <= (unsigned)CW_OWN_CAP) {
            for (unsigned e = rel; e < end; ++e) own_s[w][e] = (unsigned char)lane;
            __syncwarp();
            const unsigned char *own = own_s[w];
            cover_arcs(a, a.col + r0, total, aoff_s[w], [own](unsigned e) { return (int)own[e]; }, lane);
        } else {
            for (int i = 0; i < nm; ++i) {
                const unsigned b = __shfl_sync(0xffffffffu, rel, i), z = __shfl_sync(0xffffffffu, end, i);
                if (z - b > (unsigned)COVER_HUB) continue;  // below, in pieces
                cover_arcs(a, a.col + r0 + b, z - b, aoff_s[w], [i](unsigned) { return i; }, lane);
            }
        }
        __syncwarp();
    }
}

// The same for the hubs' rows, in pieces (apart from k_cover_walk, whose
// registers a second walk would raise).
__global__ void __launch_bounds__(CW_THREADS) k_cover_walk_hubs(CoverWalkArgs a)
{
    __shared__ int aoff_s[CW_THREADS / 32][2];
    if (*a.gate) return;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, n = *a.nhubs;
    const long long nwarps = (long long)gridDim.x * (CW_THREADS / 32);
    const long long wg = (long long)blockIdx.x * (CW_THREADS / 32) + w;
    for (int i = 0; i < n; ++i) {
        const int u = __ldg(&a.hubs[i]);
        const long long r = __ldg(&a.row_ptr[u]), end = __ldg(&a.row_ptr[u + 1]);
        if (lane < 2) aoff_s[w][lane] = __ldg(&a.off[u + lane]);
        __syncwarp();
        for (long long e0 = r + (wg + i) % nwarps * HUB_PIECE; e0 < end; e0 += nwarps * HUB_PIECE)
            cover_arcs(a, a.col + e0, (unsigned)min((long long)HUB_PIECE, end - e0), aoff_s[w],
                       [](unsigned) { return 0; }, lane);
        __syncwarp();
    }
}

// ------------------------------------------------------------------ scoring by member lists

struct CoverScoreArgs {
    const long long *row_ptr;
    const int *col;
    const int *off, *memb;     // stored-order lists
    const int *cstart, *cmem;  // members of each community
    const Rcp *recip;
    int K;
    long long E;
    int *next;                 // claim counter
    unsigned long long *g;     // GS_* accumulators
    int *status;
    const int *run_if;         // only when this flag is set (null: always)
    SmemPlan plan;             // shared-memory layout of the block
};

__global__ void __launch_bounds__(COVER_THREADS) k_cover_score(CoverScoreArgs a)
{
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ int s_c;
    if (block_stopped(a.status) || (a.run_if && !*a.run_if)) return;
    const SmemPlan &p = a.plan;
    unsigned long long *red = (unsigned long long *)(sm + p.red_off);
    int *ctl = (int *)(sm + p.ctl_off);
    unsigned long long *slot = (unsigned long long *)(sm + p.slot_off);
    int *used = (int *)(sm + p.used_off);
    const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31, wid = tid >> 5, W = T >> 5;
    for (int i = tid; i < p.cap; i += T) slot[i] = 0ull;
    if (tid < 2) ctl[tid] = 0;
    block_sync();
    const SmemTable tab{slot, used, &ctl[0], &ctl[1], p.cap, p.max_used};
    ScoreAcc acc;
    score_acc_zero(acc);
    for (;;) {
        const int c = claim_next(a.next, &s_c);
        if (c >= a.K) break;
        const int mb = __ldg(&a.cstart[c]), me = __ldg(&a.cstart[c + 1]);
        const long long size = me - mb;
        if (size == 0) continue;
        unsigned R = 1;
        for (;;) {
            unsigned long long same = 0, out = 0, slots = 0, cnt2 = 0;
            U192 pair;
            u192_zero(pair);
            bool ok = true;
            for (unsigned r = 0; r < R && ok; ++r) {
                for (int idx = mb + wid; idx < me; idx += W) {
                    const int u = __ldg(&a.cmem[idx]);
                    const int *A = a.memb + __ldg(&a.off[u]);
                    const int la = __ldg(&a.off[u + 1]) - __ldg(&a.off[u]);
                    const long long rb = __ldg(&a.row_ptr[u]), re = __ldg(&a.row_ptr[u + 1]);
                    for (long long e = rb + lane; e < re; e += 32) {
                        const int v = __ldg(&a.col[e]);
                        const int *B = a.memb + __ldg(&a.off[v]);
                        const int lb = __ldg(&a.off[v + 1]) - __ldg(&a.off[v]);
                        if (list_has(B, lb, c)) {
                            if (r == 0) ++same;
                            continue;
                        }
                        if (r == 0) ++out;
                        for (int y = 0; y < lb; ++y) {  // communities j > c that v is in and u is not
                            const int j = __ldg(&B[y]);
                            if (j <= c || list_has(A, la, j)) continue;
                            if (R == 1 || tab_split((unsigned)j, R) == r) tab_insert(tab, (unsigned)j);
                        }
                    }
                }
                block_sync();
                if (*(volatile int *)tab.overflow) {
                    ok = false;
                    break;
                }
                tab_drain(tab, tid, T, [&](int key, long long cnt) {
                    if (!QM_CHK(key, a.K, 40)) return;
                    const unsigned long long q = (unsigned long long)cnt * (unsigned long long)cnt;
                    u192_mac(pair, q, ld_rcp_cg(&a.recip[key]));
                    ++slots;
                    cnt2 += q;
                });
                block_sync();
                if (tid == 0) *tab.n_used = 0;
                block_sync();
            }
            if (!ok) {
                tab_wipe(tab, tid, T);
                block_sync();
                if (tid == 0) {
                    *tab.n_used = 0;
                    *tab.overflow = 0;
                }
                block_sync();
                if (R * 2u > R_MAX) {
                    if (tid == 0) atomicOr(a.status, 2);
                    break;
                }
                R *= 2u;
                continue;
            }
            unsigned long long w4[4] = {same, out, slots, cnt2};
            group_words_to_leader<4>(w4, T, red);
            const u128 pair_t = u192_shr64(group_u192_to_leader(pair, T, red, 128));
            if (tid == 0) {
                const long long ein = (long long)(w4[0] / 2), eout = (long long)w4[1];
                double qs, dens, contr, expn, cond;
                community_terms(ein, eout, size, a.E, qs, dens, contr, expn, cond);
                const double pen = pair_penalty_once(pair_t, size, a.E);
                const unsigned long long vol = 2ull * (unsigned long long)ein + (unsigned long long)eout;
                acc.qds_pair += fp_from_double(pen, SC_QDS);
                acc.qds_self += fp_from_double(qs, SC_QDS);
                acc.dens += fp_from_double(dens, SC_MEAN);
                acc.contr += fp_from_double(contr, SC_MEAN);
                acc.expn += fp_from_double(expn, SC_MEAN);
                acc.cond += fp_from_double(cond, SC_MEAN);
                acc.vol2 += (u128)vol * (u128)vol;
                acc.ein += (unsigned long long)ein;
                acc.eout += (unsigned long long)eout;
                acc.nonempty += 1;
                acc.slots += w4[2];
                acc.cnt2 += w4[3];
            }
            break;
        }
    }
    if (tid == 0) {  // only the leader holds sums
        limbs_add(a.g + GS_QDS_SELF, acc.qds_self);
        limbs_add(a.g + GS_QDS_PAIR, acc.qds_pair);
        limbs_add(a.g + GS_DENS, acc.dens);
        limbs_add(a.g + GS_CONTR, acc.contr);
        limbs_add(a.g + GS_EXPN, acc.expn);
        limbs_add(a.g + GS_COND, acc.cond);
        limbs_add(a.g + GS_VOL2, (i128)acc.vol2);
        const unsigned long long u[5] = {acc.ein, acc.eout, acc.nonempty, acc.slots, acc.cnt2};
        const int at[5] = {GS_EIN, GS_EOUT, GS_NONEMPTY, GS_SLOTS, GS_CNT2};
        for (int k = 0; k < 5; ++k)
            if (u[k]) atomicAdd(a.g + at[k], u[k]);
    }
}

// Eqs. (8)-(9) and the means from the sums; cut_edges_total of a cover is the
// sum over communities of |E_c^out| (an edge may leave several communities).
__global__ void k_cover_score_fin(const unsigned long long *g, const int *status, long long n, long long E,
                                  qm_quality *out)
{
    if (*status) return;
    quality_warp(g, n, E, false, out);
    __syncwarp();
    if (threadIdx.x == 0) out->cut_edges_total = (long long)g[GS_EOUT];
}

// ------------------------------------------------------------------ comparison

struct CoverCmpArgs {
    const int *aoff, *amemb, *acstart, *acmem;  // truth side
    const int *boff, *bmemb, *bcstart, *bcmem;  // found side
    const int *size_a, *size_b;
    int ka, kb;
    long long N;
    unsigned *rowmax;
    unsigned long long *rowbest;
    unsigned *colmax;
    int *next_a, *next_b, *next_c;
    unsigned long long *g;
    int *status;
    const double *logt;  // log(N / n), then n / N, 1 <= n <= LOGT_MAX (null: formed per cell)
    SmemPlan plan;
};

__device__ __forceinline__ void flush_compare_acc(const CompareAcc &acc, unsigned long long *g, unsigned long long *red)
{
    const int T = blockDim.x;
    i128 v = group_sum_i128(acc.vi, T, red);
    if (threadIdx.x == 0) limbs_add(g + GC_VI, v);
    v = group_sum_i128(acc.hnum, T, red);
    if (threadIdx.x == 0) limbs_add(g + GC_HNUM, v);
    v = group_sum_i128(acc.hden, T, red);
    if (threadIdx.x == 0) limbs_add(g + GC_HDEN, v);
    v = group_sum_i128(acc.f, T, red);
    if (threadIdx.x == 0) limbs_add(g + GC_F, v);
    const unsigned long long *src[7] = {&acc.a11, &acc.sa, &acc.sb, &acc.nvd, &acc.cells, &acc.ka, &acc.kb};
    const int dst[7] = {GC_A11, GC_SA, GC_SB, GC_NVD, GC_CELLS, GC_KA, GC_KB};
    for (int k = 0; k < 7; ++k) {
        const unsigned long long u = group_sum_u64(*src[k], T, red);
        if (threadIdx.x == 0 && u) atomicAdd(g + dst[k], u);
    }
}

// The larger of two fractions n << 32 | d (0: none), compared exactly.
__device__ __forceinline__ unsigned long long larger_fraction(unsigned long long x, unsigned long long y)
{
    if (!y) return x;
    if (!x) return y;
    return (y >> 32) * (x & 0xFFFFFFFFull) > (x >> 32) * (y & 0xFFFFFFFFull) ? y : x;
}

// The cells of every truth community a: counts |a n b| over a's members' found
// lists, then per cell the Eq. (1)-(2) terms, C(|a n b|, 2), the row's largest
// cell and F ratio (Eqs. 3-4), and each column's largest cell.
__global__ void __launch_bounds__(COVER_THREADS) k_cover_cells(CoverCmpArgs a)
{
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ int s_c;
    if (block_stopped(a.status)) return;
    const SmemPlan &p = a.plan;
    unsigned long long *red = (unsigned long long *)(sm + p.red_off);
    int *ctl = (int *)(sm + p.ctl_off);
    unsigned long long *slot = (unsigned long long *)(sm + p.slot_off);
    int *used = (int *)(sm + p.used_off);
    const int tid = threadIdx.x, T = blockDim.x;
    for (int i = tid; i < p.cap; i += T) slot[i] = 0ull;
    if (tid < 2) ctl[tid] = 0;
    block_sync();
    const SmemTable tab{slot, used, &ctl[0], &ctl[1], p.cap, p.max_used};
    CompareAcc acc;
    compare_acc_zero(acc);
    for (;;) {
        const int c = claim_next(a.next_c, &s_c);
        if (c >= a.ka) break;
        const int mb = __ldg(&a.acstart[c]), me = __ldg(&a.acstart[c + 1]);
        const long long na = me - mb;
        if (na == 0) continue;
        unsigned R = 1;
        for (;;) {
            unsigned rmax = 0;
            unsigned long long rbest = 0;  // the largest n / (n_a + n_b) as n << 32 | n_a + n_b
            CompareAcc part;
            compare_acc_zero(part);
            bool ok = true;
            for (unsigned r = 0; r < R && ok; ++r) {
                // (warp-uniform: the members of a community mostly share a found id,
                // so a warp's equal ids are merged into one update)
                for (int i0 = mb + (tid & ~31); i0 < me; i0 += T) {
                    const int idx = i0 + (tid & 31);
                    int k = 0, ke = 0;
                    if (idx < me) {
                        const int i = __ldg(&a.acmem[idx]);
                        k = __ldg(&a.boff[i]);
                        ke = __ldg(&a.boff[i + 1]);
                    }
                    while (__any_sync(0xffffffffu, k < ke)) {
                        const int b = k < ke ? __ldg(&a.bmemb[k]) : 0;
                        tab_insert_warp(tab, (unsigned)b, k < ke && (R == 1 || tab_split((unsigned)b, R) == r));
                        __syncwarp();
                        ++k;
                    }
                }
                block_sync();
                if (*(volatile int *)tab.overflow) {
                    ok = false;
                    break;
                }
                tab_drain(tab, tid, T, [&](int b, long long n) {
                    if (!QM_CHK(b, a.kb, 41)) return;
                    const long long nb = __ldg(&a.size_b[b]);
                    part.a11 += (unsigned long long)(n * (n - 1) / 2);
                    part.cells += 1;
                    const double l1 = cell_log(n, na, nb);
                    part.vi += fp_from_double(vi_term_l(n, l1), SC_VI);
                    const bool tb = a.logt && n <= LOGT_MAX;
                    part.hnum += fp_from_double(nmi_num_term_q(tb ? __ldg(&a.logt[LOGT_MAX + 1 + n]) : nmi_over(n, a.N), l1,
                                                               tb ? __ldg(&a.logt[n]) : log_ratio(a.N, n)),
                                                SC_H);
                    rmax = max(rmax, (unsigned)n);
                    rbest = larger_fraction(rbest, ((unsigned long long)n << 32) | (unsigned long long)(na + nb));
                    atomicMax(&a.colmax[b], (unsigned)n);
                });
                block_sync();
                if (tid == 0) *tab.n_used = 0;
                block_sync();
            }
            if (!ok) {
                tab_wipe(tab, tid, T);
                block_sync();
                if (tid == 0) {
                    *tab.n_used = 0;
                    *tab.overflow = 0;
                }
                block_sync();
                if (R * 2u > R_MAX) {
                    if (tid == 0) atomicOr(a.status, 2);
                    break;
                }
                R *= 2u;
                continue;
            }
            compare_acc_add(acc, part);
            // the row's largest cell and ratio (divided once: rounding is monotone,
            // so the largest rounded ratio is the rounded largest ratio)
            const unsigned m = group_max_u32(rmax, T, red);
            unsigned long long bb = rbest;
            for (int d = 16; d > 0; d >>= 1) bb = larger_fraction(bb, __shfl_down_sync(0xffffffffu, bb, d));
            block_sync();
            if ((tid & 31) == 0) red[tid >> 5] = bb;
            block_sync();
            if (tid == 0) {
                unsigned long long best = 0;
                for (int w = 0; w < (T >> 5); ++w) best = larger_fraction(best, red[w]);
                a.rowmax[c] = m;
                const long long bn = (long long)(best >> 32), bd = (long long)(best & 0xFFFFFFFFull);
                a.rowbest[c] = bn ? (unsigned long long)__double_as_longlong(f_ratio(bn, na, bd - na)) : 0ull;
            }
            break;
        }
    }
    flush_compare_acc(acc, a.g, red);
}

// Row side (truth communities): C(|a|, 2), the entropy term, F, NVD row maxima.
__global__ void k_cover_rows(CoverCmpArgs a)
{
    __shared__ unsigned long long red[72];
    if (*a.status) return;
    CompareAcc acc;
    compare_acc_zero(acc);
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < a.ka; c += gridDim.x * blockDim.x) {
        const long long na = a.size_a[c];
        if (na == 0) continue;
        acc.sa += (unsigned long long)(na * (na - 1) / 2);
        acc.nvd += a.rowmax[c];
        acc.f += fp_from_double(__dmul_rn((double)na, __longlong_as_double((long long)a.rowbest[c])), SC_F);
        acc.hden += fp_from_double(entropy_term(na, a.N), SC_H);
        acc.ka += 1;
    }
    flush_compare_acc(acc, a.g, red);
}

// Column side (found communities): C(|b|, 2), the entropy term, NVD column maxima.
__global__ void k_cover_cols(CoverCmpArgs a)
{
    __shared__ unsigned long long red[72];
    if (*a.status) return;
    CompareAcc acc;
    compare_acc_zero(acc);
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < a.kb; c += gridDim.x * blockDim.x) {
        const long long nb = a.size_b[c];
        if (nb == 0) continue;
        acc.sb += (unsigned long long)(nb * (nb - 1) / 2);
        acc.nvd += a.colmax[c];
        acc.hden += fp_from_double(entropy_term(nb, a.N), SC_H);
        acc.kb += 1;
    }
    flush_compare_acc(acc, a.g, red);
}

// Pair-count corrections for pairs of nodes sharing two or more communities on
// side X (the other side is Y).  For community c of X, its members with two or
// more memberships are paired up; a pair is taken by the smallest community
// the two share in X, so once.  With k = |X(i) n X(j)| and k' = |Y(i) n Y(j)|:
//   same_X correction  k - 1                      (when k >= 2)
//   a11 correction     k k' - 1 (side A, k >= 2, k k' >= 1), or k' - 1 (side B,
//                      k' >= 2 and k = 1, the pairs side A did not take)
template <bool SIDE_A>
__global__ void __launch_bounds__(COVER_THREADS) k_cover_pairs(CoverCmpArgs a)
{
    __shared__ int s_c, s_n;
    __shared__ int ovl[OVL_CAP];
    __shared__ unsigned long long red[72];
    if (*a.status) return;
    const int *xoff = SIDE_A ? a.aoff : a.boff, *xmemb = SIDE_A ? a.amemb : a.bmemb;
    const int *yoff = SIDE_A ? a.boff : a.aoff, *ymemb = SIDE_A ? a.bmemb : a.amemb;
    const int *xcstart = SIDE_A ? a.acstart : a.bcstart, *xcmem = SIDE_A ? a.acmem : a.bcmem;
    const int kx = SIDE_A ? a.ka : a.kb;
    const int tid = threadIdx.x, T = blockDim.x;
    unsigned long long same_corr = 0, a11_corr = 0;
    for (;;) {
        const int c = claim_next(SIDE_A ? a.next_a : a.next_b, &s_c);
        if (c >= kx) break;
        const int mb = __ldg(&xcstart[c]), me = __ldg(&xcstart[c + 1]);
        if (me - mb < 2) continue;
        // members with two or more memberships on this side
        if (tid == 0) s_n = 0;
        block_sync();
        for (int idx = mb + tid; idx < me; idx += T) {
            const int i = __ldg(&xcmem[idx]);
            if (__ldg(&xoff[i + 1]) - __ldg(&xoff[i]) >= 2) {
                const int at = atomicAdd(&s_n, 1);
                if (at < OVL_CAP) ovl[at] = i;
            }
        }
        block_sync();
        const int L = s_n;
        if (L < 2) continue;
        const bool in_smem = L <= OVL_CAP;
        // pairs of overlapping members (from shared memory, or the whole member
        // list filtered again when there are too many to hold)
        // The pairs (p, q), p < q < Lp, as a rectangle: with Lp rounded up to an even
        // number E, rows p and E - 1 - p hold E - 1 pairs together, so E / 2 rows of
        // E - 1 columns hold all (those with q = Lp are none where Lp is odd).  Every
        // thread steps through it T places at a time, without a division a pair.
        const unsigned Lp = in_smem ? L : me - mb, E = Lp + (Lp & 1u), width = E - 1u;
        const unsigned dr = T / width, dq = T % width;
        unsigned row = tid / width, at = tid % width;
        for (; row < E / 2u; row += dr, at += dq, row += at >= width ? 1u : 0u, at -= at >= width ? width : 0u) {
            const bool upper = at >= row;
            const unsigned pp = upper ? row : E - 1u - row, qq = upper ? at + 1u : E - row + at;
            if (qq >= Lp) continue;
            const int i = in_smem ? ovl[pp] : __ldg(&xcmem[mb + pp]);
            const int j = in_smem ? ovl[qq] : __ldg(&xcmem[mb + qq]);
            const int li = __ldg(&xoff[i + 1]) - __ldg(&xoff[i]), lj = __ldg(&xoff[j + 1]) - __ldg(&xoff[j]);
            if (li < 2 || lj < 2) continue;
            int first = 0, dummy = 0;
            const int kxx = list_meet(xmemb + __ldg(&xoff[i]), li, xmemb + __ldg(&xoff[j]), lj, &first);
            if (first != c || kxx < 2) continue;
            const int kyy = list_meet(ymemb + __ldg(&yoff[i]), __ldg(&yoff[i + 1]) - __ldg(&yoff[i]),
                                      ymemb + __ldg(&yoff[j]), __ldg(&yoff[j + 1]) - __ldg(&yoff[j]), &dummy);
            same_corr += (unsigned long long)(kxx - 1);
            if (SIDE_A) {
                if (kyy >= 1) a11_corr += (unsigned long long)(kxx * kyy - 1);
            } else {
                if (kyy == 1) a11_corr += (unsigned long long)(kxx - 1);
            }
        }
    }
    const unsigned long long s = group_sum_u64(same_corr, T, red);
    const unsigned long long q = group_sum_u64(a11_corr, T, red);
    if (tid == 0) {
        if (s) atomicAdd(a.g + (SIDE_A ? GC_SAME_A_CORR : GC_SAME_B_CORR), s);
        if (q) atomicAdd(a.g + GC_A11_CORR, q);
    }
}

__global__ void k_cover_compare_fin(const unsigned long long *g, const int *status, long long n, qm_compare *out)
{
    __shared__ unsigned long long w[GC_COUNT];
    if (*status) return;
    const int lane = threadIdx.x;
    if (lane < GC_COUNT)
        w[lane] = g[lane] - (lane == GC_A11 ? g[GC_A11_CORR] : lane == GC_SA ? g[GC_SAME_A_CORR]
                             : lane == GC_SB ? g[GC_SAME_B_CORR] : 0ull);
    __syncwarp();
    compare_warp(w, n, out);
}

// ------------------------------------------------------------------ launchers

namespace {

int grid_of(long long n, int threads, int num_sms, int per_sm)
{
    long long g = (n + threads - 1) / threads;
    g = std::min<long long>(g, (long long)num_sms * per_sm);
    return (int)std::max<long long>(g, 1);
}

// Member lists of a cover's communities (run_if: only when that flag is set).
int members_of_side(const CoverSide &c, long long n, const CoverWs &w, int num_sms, cudaStream_t s, const int *run_if)
{
    const int l2 = scan_offsets(c.size, c.K, c.cstart, w.scan_tmp, w.counters + CC_SCAN, w.status, s);
    if (l2 < 0) return -1;
    k_cover_scatter<<<grid_of(n, 256, num_sms, 8), 256, 0, s>>>(c.off, c.memb, n, c.cstart, c.cur, c.cmem, w.status,
                                                               run_if);
    return l2 + 1;
}

// Brings one cover to the stored order and builds its member lists (members).
int prepare_side(const long long *mptr, const int *memb, long long m, long long n, const int *inv,
                 const CoverSide &c, const CoverWs &w, int num_sms, cudaStream_t s, int *head = nullptr,
                 int *too_long = nullptr, const long long *row_ptr = nullptr, bool members = true)
{
    int L = 0;
    k_cover_len<<<grid_of(n, 256, num_sms, 8), 256, 0, s>>>(mptr, n, m, inv, c.len, w.status, too_long);
    ++L;
    const int l1 = scan_offsets(c.len, (int)n, c.off, w.scan_tmp, w.counters + CC_SCAN, w.status, s);
    if (l1 < 0) return -1;
    L += l1;
    k_cover_copy<<<grid_of(n, 256, num_sms, 8), 256, 0, s>>>(mptr, memb, n, inv, c.K, c.off, c.memb, c.size,
                                                            w.status, head, row_ptr, w.hubs, w.counters + CC_HUBS);
    ++L;
    if (!members) return L;
    const int l2 = members_of_side(c, n, w, num_sms, s, nullptr);
    return l2 < 0 ? -1 : L + l2;
}

}  // namespace

void prepare_cover_kernels()
{
    cudaFuncSetAttribute(k_cover_score, cudaFuncAttributeMaxDynamicSharedMemorySize, COVER_SMEM);
    cudaFuncSetAttribute(k_cover_cells, cudaFuncAttributeMaxDynamicSharedMemorySize, COVER_SMEM);
    k_fill_log_int<<<(LOGT_MAX + 256) / 256, 256>>>();  // this unit's copy of the log(i) table
    cudaDeviceSynchronize();
}

int launch_cover_score(const GraphDev &g, const long long *mptr, const int *memb, long long m, int K,
                       const CoverWs &w, int num_sms, cudaStream_t s)
{
    const long long n = g.n;
    const bool runs = w.run_entries > 0;
    int L = prepare_side(mptr, memb, m, n, g.inv, w.a, w, num_sms, s, runs ? w.head : nullptr,
                         runs ? w.counters + CC_LONG : nullptr, g.row_ptr, !runs);
    if (L < 0) return -1;
    const int *run_if = nullptr;
    if (runs) {
        int *const gate = w.counters + CC_GATE, *const old_path = w.counters + CC_OLD;
        unsigned long long *const total = (unsigned long long *)(w.counters + CC_TOTAL);
        k_cover_cap<<<grid_of(n, 256, num_sms, 8), 256, 0, s>>>(g.row_ptr, g.col, w.a.off, w.a.memb, w.head, n, w.cv, w.capw,
                                                               total, w.hubs, w.counters + CC_HUBS,
                                                               w.counters + CC_LONG, w.status);
        k_cover_gate<<<1, 1, 0, s>>>(w.status, total, w.run_entries, w.counters + CC_LONG, gate, old_path);
        L += 2 + launch_segment_bases(w.capw, K, w.base, w.recip, (unsigned *)w.scan_tmp, gate, s);
        CoverWalkArgs a;
        a.row_ptr = g.row_ptr;
        a.col = g.col;
        a.off = w.a.off;
        a.memb = w.a.memb;
        a.head = w.head;
        a.n = n;
        a.base = w.base;
        a.curs = w.curs;
        a.nbr = w.nbr;
        a.hubs = w.hubs;
        a.nhubs = w.counters + CC_HUBS;
        a.gate = gate;
        k_cover_walk<<<grid_of(n, CW_THREADS, num_sms, 5), CW_THREADS, 0, s>>>(a);
        k_cover_walk_hubs<<<5 * num_sms, CW_THREADS, 0, s>>>(a);
        CoverRuns r;
        r.cv = w.cv;
        r.curs = w.curs;
        r.base = w.base;
        r.nbr = w.nbr;
        r.recip = w.recip;
        r.inter = w.inter;
        r.rec = w.rec;
        for (int k = 0; k < 4; ++k) r.hdr[k] = w.hdr[k];
        r.counters = w.counters + CC_RUNS;
        r.gate = gate;
        r.err = w.status;
        const int lr = launch_cover_runs(r, K, g.n_arcs / 2, w.gacc, num_sms, s);
        if (lr < 0) return -1;
        L += 2 + lr;
        run_if = old_path;  // the kernels below work only when the runs did not fit
        const int lm = members_of_side(w.a, n, w, num_sms, s, run_if);
        if (lm < 0) return -1;
        L += lm;
    }
    k_cover_rcp<<<grid_of(K, 256, num_sms, 4), 256, 0, s>>>(w.a.size, K, w.recip, w.status, run_if);
    CoverScoreArgs a;
    a.row_ptr = g.row_ptr;
    a.col = g.col;
    a.off = w.a.off;
    a.memb = w.a.memb;
    a.cstart = w.a.cstart;
    a.cmem = w.a.cmem;
    a.recip = w.recip;
    a.K = K;
    a.E = g.n_arcs / 2;
    a.next = w.counters + CC_NEXT_C;
    a.g = w.gacc;
    a.status = w.status;
    a.run_if = run_if;
    a.plan = plan_smem(COVER_THREADS, COVER_SMEM);
    k_cover_score<<<std::min(num_sms * 4, std::max(K, 1)), COVER_THREADS, COVER_SMEM, s>>>(a);
    k_cover_score_fin<<<1, 32, 0, s>>>(w.gacc, w.status, n, g.n_arcs / 2, (qm_quality *)w.result);
    L += 3;
    return cudaGetLastError() == cudaSuccess ? L : -1;
}

int launch_cover_compare(const long long *aptr, const int *amemb, long long ma, int ka, const long long *bptr,
                         const int *bmemb, long long mb, int kb, long long n, const CoverWs &w, int num_sms,
                         cudaStream_t s)
{
    int L1 = prepare_side(aptr, amemb, ma, n, nullptr, w.a, w, num_sms, s);
    if (L1 < 0) return -1;
    int L2 = prepare_side(bptr, bmemb, mb, n, nullptr, w.b, w, num_sms, s);
    if (L2 < 0) return -1;
    CoverCmpArgs a;
    a.aoff = w.a.off;
    a.amemb = w.a.memb;
    a.acstart = w.a.cstart;
    a.acmem = w.a.cmem;
    a.boff = w.b.off;
    a.bmemb = w.b.memb;
    a.bcstart = w.b.cstart;
    a.bcmem = w.b.cmem;
    a.size_a = w.a.size;
    a.size_b = w.b.size;
    a.ka = ka;
    a.kb = kb;
    a.N = n;
    a.rowmax = w.rowmax;
    a.rowbest = w.rowbest;
    a.colmax = w.colmax;
    a.next_a = w.counters + CC_NEXT_A;
    a.next_b = w.counters + CC_NEXT_B;
    a.next_c = w.counters + CC_NEXT_C;
    a.g = w.gacc;
    a.status = w.status;
    // the tables are a launch more, which few cells do not repay (10^3 nodes in
    // one community each: 207 us a call with them, 192 without)
    const bool tables = ma + mb > COVER_TABLE_MEMB;
    a.logt = tables ? w.logt : nullptr;
    a.plan = plan_smem(COVER_THREADS, COVER_SMEM);
    if (tables) launch_batch_logt(w.logt, n, s);
    k_cover_cells<<<std::min(num_sms * 4, std::max(ka, 1)), COVER_THREADS, COVER_SMEM, s>>>(a);
    k_cover_rows<<<grid_of(ka, 256, num_sms, 2), 256, 0, s>>>(a);
    k_cover_cols<<<grid_of(kb, 256, num_sms, 2), 256, 0, s>>>(a);
    k_cover_pairs<true><<<std::min(num_sms * 4, std::max(ka, 1)), COVER_THREADS, 0, s>>>(a);
    k_cover_pairs<false><<<std::min(num_sms * 4, std::max(kb, 1)), COVER_THREADS, 0, s>>>(a);
    k_cover_compare_fin<<<1, 32, 0, s>>>(w.gacc, w.status, n, (qm_compare *)w.result);
    return cudaGetLastError() == cudaSuccess ? L1 + L2 + 6 + (tables ? 1 : 0) : -1;
}

}  // namespace qm
