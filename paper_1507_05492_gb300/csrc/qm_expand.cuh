// qm_expand.cuh -- parts of phase A of the two-phase scoring pipeline (the
// far-end label gathers): the label encodings, the gathers in community order of
// the batched pipeline (qm_batched.cu) and of the half-edge variant
// (qm_kernels.cu).  The single-partition default, in node order, is in qm_rows.cuh.
#pragma once

#include <climits>

#include "qm_community.cuh"

namespace qm {
using namespace qmk;

// Phase A in community order: for each member position p the labels of the
// neighbours of members[p] are looked up.  A warp takes 32 consecutive member
// positions; they hold one or more runs of members of one community each.  For
// a run of community c the warp spreads the run's arcs over its lanes,
// gathers the neighbour labels, and packs those != c at the front of c's arc
// segment: a ballot gives each lane its place and one atomic on inter[c]
// reserves the room.  inter[c] ends as the number of cut arcs of c,
// |E_c^out| (Sec. II-B.3), and the packed run never outgrows the segment,
// whose length is the volume of c.  No shared-memory table is needed, so the
// kernel runs at full occupancy.
//
// Locating the CSR entry of the e-th arc of a run: when the 32 members form a
// few segments of consecutive node ids (the common case on a graph loaded
// with QM_REORDER), a segment's rows are adjacent in the CSR and its arcs are
// one contiguous range; otherwise a search over the members' arc offsets
// finds the member of each arc.
constexpr int EXPAND_THREADS = 256;

// Community ownership of a sharded call (the decomposition of Sec. III-A:
// community c belongs to process c mod P).  Unsharded calls pass P = 1.
struct Shard {
    int r;  // this shard
    int p;  // number of shards
    __device__ __forceinline__ bool owns(int c) const { return p == 1 || c % p == r; }
};
constexpr int EXPAND_UNROLL = 8;
constexpr int EXPAND_MAX_SEGS = 6;

// Edge weights of a weighted graph (float32, 0 or in [2^-20, 2^20)) as exact
// fixed-point integers: w * 2^43 (an integer below 2^63).
__device__ __forceinline__ unsigned long long w_fixed(float w) { return __float2ull_rn(w * 8796093022208.0f); }

// Packed copy of the labels for the far-end gathers: three 21-bit labels per
// 64-bit word (label ids below 2^21), 8/3 bytes a node instead of 4.  The
// gathers of the expand phase land at random in the label array; a smaller
// array leaves a larger share of it in L2.
constexpr int PACK_BITS = 21;
constexpr long long PACK_MAX_K = 1LL << PACK_BITS;

__device__ __forceinline__ int ld_label3(const unsigned long long *plab, int v, unsigned long long pol)
{
    const unsigned q = (unsigned)v / 3u;
    const unsigned r = (unsigned)v - 3u * q;
    unsigned long long w;
    asm("ld.global.nc.L2::cache_hint.b64 %0, [%1], %2;" : "=l"(w) : "l"(plab + q), "l"(pol));
    return (int)((w >> (PACK_BITS * r)) & 0x1FFFFFull);
}

// Block encoding of the labels of a renumbered graph, for the far-end gathers
// (built per call by k_pack_blocks).  Along the stored node order the labels
// of a partition that follows the graph's clusters change rarely, so most
// blocks of 16 consecutive nodes carry one label: one 32-bit word per block
// holds it.  A block of two labels has its word point (BLK_PAIR) at a 64-bit
// entry with labels A ([0, 21)) and B ([21, 42)) and a 16-bit mask that selects
// B; a block of more at a slot of its 16 labels (BLK_SLOT).  The words of 10^8
// nodes take 25 MB (the packed copy 267 MB), so the encoding stays in L2, and
// most gathers are one 32-bit load and a sign test.
constexpr int BLK_NODES = 16;
constexpr unsigned BLK_SLOT = 0x80000000u, BLK_PAIR = 0xC0000000u, BLK_INDEX = 0x3FFFFFFFu;

// Where the pairs and the slots begin, in 32-bit words from the array's start.
__host__ __device__ inline unsigned blk_pairs_at(long long n)
{
    return (unsigned)(((n + BLK_NODES - 1) / BLK_NODES + 31) / 32 * 32);
}
__host__ __device__ inline unsigned blk_slots_at(long long n) { return 3u * blk_pairs_at(n); }

// Label sources of the far-end gathers: the labels as given, the packed copy,
// or the block encoding.
enum { LAB_PLAIN = 0, LAB_PACK3 = 1, LAB_BLOCKS = 2 };

// Gathers the labels of arcs [e_lo, e_hi) of a run of community c (loc(e) is
// the CSR index of arc e), counts those != c in inter[c] (the cut arcs of c)
// and packs those above c into c's segment at cbase (each unordered pair of
// communities is counted by its smaller id); hi[c] counts them.
template <class LOC>
__device__ __forceinline__ void expand_range(unsigned e_lo, unsigned e_hi, int c, unsigned cbase, LOC loc,
                                             const int *__restrict__ col, const int *__restrict__ labels,
                                             int *inter, int *hi, int *__restrict__ nbr, unsigned long long keep,
                                             int lane)
{
    const unsigned lt = (1u << lane) - 1u;
    for (unsigned e0 = e_lo; e0 < e_hi; e0 += 32u * EXPAND_UNROLL) {
        int lab[EXPAND_UNROLL];
#pragma unroll
        for (int k = 0; k < EXPAND_UNROLL; ++k) {
            const unsigned e = e0 + lane + 32u * k;
            lab[k] = e < e_hi ? __ldcs(&col[loc(e)]) : -1;
        }
#pragma unroll
        for (int k = 0; k < EXPAND_UNROLL; ++k)
            if (lab[k] >= 0) lab[k] = ld_hint(&labels[lab[k]], keep);
        unsigned msk[EXPAND_UNROLL];
        int tot = 0, cut = 0;
#pragma unroll
        for (int k = 0; k < EXPAND_UNROLL; ++k) {
            cut += __popc(__ballot_sync(0xffffffffu, lab[k] >= 0 && lab[k] != c));
            msk[k] = __ballot_sync(0xffffffffu, lab[k] > c);
            tot += __popc(msk[k]);
        }
        if (cut && lane == 0) atomicAdd(&inter[c], cut);
        if (tot == 0) continue;
        int pos = 0;
        if (lane == 0) pos = atomicAdd(&hi[c], tot);
        unsigned at = cbase + (unsigned)__shfl_sync(0xffffffffu, pos, 0);
#pragma unroll
        for (int k = 0; k < EXPAND_UNROLL; ++k) {
            if ((msk[k] >> lane) & 1u) __stcs(&nbr[at + __popc(msk[k] & lt)], lab[k]);
            at += __popc(msk[k]);
        }
    }
}

// Warp total of lane sums of fixed-point weights: four 27-bit chunks, each added
// by one redux.  A lane holds a 32nd of the arcs of a stretch of rows, fewer than
// 2^27 weights below 2^63, so its sum is below 2^90.
__device__ __forceinline__ u128 warp_sum_u108(u128 v)
{
    constexpr unsigned M = (1u << 27) - 1u;
    u128 r = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) r += (u128)__reduce_add_sync(0xffffffffu, (unsigned)(v >> (27 * k)) & M) << (27 * k);
    return r;
}

// A community's sum of fixed-point weights in global memory: v = L2 * 2^64 +
// L1 * 2^32 + L0, updated with 64-bit atomics, where L0 and L1 add up 32-bit
// chunks and L2 the rest.  Every addition brings at least one arc, of which there
// are fewer than 2^32, each below 2^63: no word passes 2^64, however a community's
// nodes lie (limbs_add holds only 2^21 additions).
__device__ __forceinline__ void wsum_add(unsigned long long *L, u128 v)
{
    const unsigned long long l0 = (unsigned)v, l1 = (unsigned)(v >> 32), l2 = (unsigned long long)(v >> 64);
    if (l0) atomicAdd(&L[0], l0);
    if (l1) atomicAdd(&L[1], l1);
    if (l2) atomicAdd(&L[2], l2);
}

__device__ __forceinline__ i128 wsum_get(const unsigned long long *L)
{
    return (i128)(((u128)L[2] << 64) + ((u128)L[1] << 32) + (u128)L[0]);
}

// The same sum below 2^96 in three 32-bit words of shared memory, the carries
// passed on by whoever causes them.
__device__ __forceinline__ void wsum_add_smem(unsigned *L, u128 v)
{
    const unsigned l0 = (unsigned)v;
    unsigned carry = l0 && atomicAdd(&L[0], l0) > ~l0 ? 1u : 0u;
    const unsigned l1 = (unsigned)(v >> 32) + carry;
    if (l1) carry = atomicAdd(&L[1], l1) > ~l1 ? 1u : 0u;  // (else the carry, if any, went through l1)
    const unsigned l2 = (unsigned)(v >> 64) + carry;
    if (l2) atomicAdd(&L[2], l2);
}

// Where a kernel adds up the communities' weights: six words per community,
// intra then cut, in global memory, or (few communities) in a block's shared
// memory, whose sums it adds to the global ones at its end.
struct WeightSums {
    unsigned long long *wl;
    unsigned *smem;  // null: straight to wl

    __device__ __forceinline__ void add(int c, u128 w_in, u128 w_out) const
    {
        if (smem) {
            if (w_in) wsum_add_smem(smem + c * 6, w_in);
            if (w_out) wsum_add_smem(smem + c * 6 + 3, w_out);
        } else {
            if (w_in) wsum_add(wl + (size_t)c * 6, w_in);
            if (w_out) wsum_add(wl + (size_t)c * 6 + 3, w_out);
        }
    }
};

// Adds a warp's intra and cut weight sums of community c.
__device__ __forceinline__ void flush_weights(const WeightSums &ws, int c, u128 w_in, u128 w_out, int lane)
{
    w_in = warp_sum_u108(w_in);
    w_out = warp_sum_u108(w_out);
    if (lane == 0) ws.add(c, w_in, w_out);
}

// ---------------------------------------------------------------- half-edge gathers
//
// On a graph that also holds its upper rows (each node's arcs to itself and to
// higher node ids, a self-loop stored as ~u), every undirected edge is gathered
// once, from its lower end.  An arc of a member of c to community l != c puts
// one entry into the run of the smaller of the two ids: l packed into c's
// segment when l > c, c appended to l's segment (through l's run cursor and
// segment base cbase[l]) when l < c; with FULL both.  Arcs inside c add 2 (a
// self-loop 1) to same2[c], so E_c^out = vol(c) - same2[c] and the runs hold the
// same multisets as gathering every arc from both ends.
template <bool PACK, bool FULL, class LOC>
__device__ __forceinline__ void expand_range_half(unsigned e_lo, unsigned e_hi, int c, unsigned cbase_c, LOC loc,
                                                  const int *__restrict__ up_col, const int *__restrict__ labels,
                                                  const unsigned long long *__restrict__ plab, int *same2,
                                                  int *cursor, const unsigned *__restrict__ cbase,
                                                  int *__restrict__ nbr, unsigned long long keep, int lane)
{
    const unsigned lt = (1u << lane) - 1u;
    for (unsigned e0 = e_lo; e0 < e_hi; e0 += 32u * EXPAND_UNROLL) {
        int lab[EXPAND_UNROLL];
        unsigned intra = 0;
#pragma unroll
        for (int k = 0; k < EXPAND_UNROLL; ++k) {
            const unsigned e = e0 + lane + 32u * k;
            lab[k] = e < e_hi ? __ldcs(&up_col[loc(e)]) : INT_MIN;
        }
#pragma unroll
        for (int k = 0; k < EXPAND_UNROLL; ++k) {
            if (lab[k] == INT_MIN) {
                lab[k] = -1;
            } else if (lab[k] < 0) {  // a self-loop: one arc inside c
                intra += 1u;
                lab[k] = -1;
            } else {
                lab[k] = PACK ? ld_label3(plab, lab[k], keep) : ld_hint(&labels[lab[k]], keep);
                if (lab[k] == c) {
                    intra += 2u;
                    lab[k] = -1;
                }
            }
        }
        intra = __reduce_add_sync(0xffffffffu, intra);
        if (intra && lane == 0) atomicAdd(&same2[c], (int)intra);
        // entries for c's own run
        unsigned msk[EXPAND_UNROLL];
        int tot = 0;
#pragma unroll
        for (int k = 0; k < EXPAND_UNROLL; ++k) {
            msk[k] = __ballot_sync(0xffffffffu, FULL ? lab[k] >= 0 : lab[k] > c);
            tot += __popc(msk[k]);
        }
        if (tot) {
            int pos = 0;
            if (lane == 0) pos = atomicAdd(&cursor[c], tot);
            unsigned at = cbase_c + (unsigned)__shfl_sync(0xffffffffu, pos, 0);
#pragma unroll
            for (int k = 0; k < EXPAND_UNROLL; ++k) {
                if ((msk[k] >> lane) & 1u) __stcs(&nbr[at + __popc(msk[k] & lt)], lab[k]);
                at += __popc(msk[k]);
            }
        }
        // c appended to the runs of the smaller neighbouring ids (FULL: all),
        // lanes of one destination merged into one cursor update; all cursor
        // updates and segment bases of the step are in flight at once
        unsigned peers[EXPAND_UNROLL];
        int base[EXPAND_UNROLL];
        unsigned cb[EXPAND_UNROLL];
#pragma unroll
        for (int k = 0; k < EXPAND_UNROLL; ++k) {
            const bool rem = FULL ? lab[k] >= 0 : (lab[k] >= 0 && lab[k] < c);
            const unsigned rm = __ballot_sync(0xffffffffu, rem);
            peers[k] = rem ? __match_any_sync(rm, lab[k]) : 0u;
        }
#pragma unroll
        for (int k = 0; k < EXPAND_UNROLL; ++k) {
            base[k] = 0;
            if (peers[k] && lane == __ffs(peers[k]) - 1) base[k] = atomicAdd(&cursor[lab[k]], __popc(peers[k]));
            if (peers[k]) cb[k] = __ldg(&cbase[lab[k]]);
        }
#pragma unroll
        for (int k = 0; k < EXPAND_UNROLL; ++k) {
            if (!peers[k]) continue;
            const int b = __shfl_sync(peers[k], base[k], __ffs(peers[k]) - 1);
            nbr[cb[k] + (unsigned)(b + __popc(peers[k] & lt))] = c;
        }
    }
}

// One warp's share of the half-edge phase A: 32 member positions, over the
// members' upper rows (up_ptr / up_col), with the in-chunk arc offsets summed
// in the warp and each community's segment base read from cbase.
template <bool PACK, bool FULL>
__device__ __forceinline__ void expand_chunk_half(long long p0, long long n, const long long *__restrict__ up_ptr,
                                                  const int *__restrict__ up_col, const int *__restrict__ labels,
                                                  const unsigned long long *__restrict__ plab,
                                                  const int *__restrict__ members, const unsigned *__restrict__ cbase,
                                                  int *same2, int *cursor, int *__restrict__ nbr, unsigned *offw,
                                                  long long *rsw, int *cw, unsigned long long keep, int lane)
{
    const int nm = (int)min(32LL, n - p0);
    int u = -2;
    unsigned d = 0;
    if (lane < nm) {
        u = __ldcs(&members[p0 + lane]);
        rsw[lane] = __ldg(&up_ptr[u]);
        d = (unsigned)(__ldg(&up_ptr[u + 1]) - rsw[lane]);
        cw[lane] = ld_hint(&labels[u], keep);
    }
    unsigned inc = d;
#pragma unroll
    for (int s2 = 1; s2 < 32; s2 <<= 1) {
        const unsigned t = __shfl_up_sync(0xffffffffu, inc, s2);
        if (lane >= s2) inc += t;
    }
    if (lane < nm) offw[lane] = inc - d;
    if (lane == nm - 1) offw[nm] = inc;
    __syncwarp();
    const int u_prev = __shfl_up_sync(0xffffffffu, u, 1);
    const bool valid = lane < nm;
    const bool newrun = valid && (lane == 0 || cw[lane] != cw[lane - 1]);
    unsigned runs = __ballot_sync(0xffffffffu, newrun);
    const unsigned segs = __ballot_sync(0xffffffffu, newrun || (valid && u != u_prev + 1));
    if (__popc(segs) <= EXPAND_MAX_SEGS) {
        unsigned rem = segs;
        while (rem) {
            const int lo = __ffs(rem) - 1;
            rem &= rem - 1;
            const int hi = rem ? __ffs(rem) - 1 : nm;
            const unsigned e_lo = offw[lo], e_hi = offw[hi];
            if (e_lo == e_hi) continue;
            const int c = cw[lo];
            const long long cs = rsw[lo] - (long long)e_lo;  // upper-row index of arc e is cs + e
            expand_range_half<PACK, FULL>(e_lo, e_hi, c, __ldg(&cbase[c]),
                                          [cs](unsigned e) { return cs + (long long)e; }, up_col, labels, plab,
                                          same2, cursor, cbase, nbr, keep, lane);
        }
    } else {
        while (runs) {
            const int m_lo = __ffs(runs) - 1;
            runs &= runs - 1;
            const int m_hi = runs ? __ffs(runs) - 1 : nm;
            const unsigned e_lo = offw[m_lo], e_hi = offw[m_hi];
            if (e_lo == e_hi) continue;
            const int c = cw[m_lo];
            expand_range_half<PACK, FULL>(
                e_lo, e_hi, c, __ldg(&cbase[c]),
                [=](unsigned e) {
                    const int o = m_lo + upper_bound_smem(offw + m_lo, m_hi - m_lo, e) - 1;
                    return rsw[o] + (long long)(e - offw[o]);
                },
                up_col, labels, plab, same2, cursor, cbase, nbr, keep, lane);
        }
    }
    __syncwarp();
}

}  // namespace qm
