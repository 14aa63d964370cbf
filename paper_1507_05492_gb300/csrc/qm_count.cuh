// qm_count.cuh -- phase B of the two-phase scoring pipeline with one-word counting
// tables: |E_ci,cj| (Eq. (9)) of every neighbour of a community from its packed run.
//
// What a run needs is T_c = sum_j |E_cj|^2 Rcp_j over its distinct keys j.  With
// the occurrences of a key numbered 1, 2, ..., the k-th adds (2k - 1) Rcp_j, so
// every entry adds Rcp_j once whatever the table says, and only a repeat adds
// more: 2 Rcp_j times the occurrences before it.  The table therefore holds one
// 32-bit word a slot, the key (+1) above and its repeats so far in the low `cb`
// bits, 0 for a free slot: an entry is one compare-and-swap at its hash (free:
// first occurrence; own key: one add returns its number; else the next slot).
// Runs are at most 3/4 of the slots they hash into and shorter than 2^cb, so a
// free slot is always found and no count can reach the key's bits.
//
// What bounds it and why this shape: the pass moves few bytes (a run's labels
// once, 16 bytes of reciprocal a key from L2); it is bound by instructions and
// shared-memory atomics.  So each lane keeps CT_UNROLL entries in flight (all
// their compare-and-swaps are issued before any is looked at, and the
// reciprocals arrive meanwhile), and the entries whose first slot was taken
// (about a fifth) are not followed by the lanes that met them, which would
// keep the others waiting for the longest chain, but collected in shared
// memory and followed 32 at a time.  The table of a run is a power of two
// sized by the run (cleared afterwards with 16-byte stores), which lets 32
// warps share an SM's shared memory and leaves L1 room for the loads in flight
// (tables of twice the size: 1.13 against 0.66 ms for k_count_tab at 3.2*10^7
// nodes; ten or twelve blocks an SM at fewer registers: 0.69-1.13 ms).
//
// Measured, k_count_tab + k_count_big against k_count + k_count_long (tables of
// two words a slot, a lane following its own chains): 10^8 nodes, planted,
// 3.3*10^8 entries: 2.85 against 4.02 ms; 10^7 nodes with 20% moved: 0.51
// against 1.61 ms; 10^6 nodes, every label counted: 0.15 against 0.41 ms.
#pragma once

#include <type_traits>

#include "qm_community.cuh"

namespace qmk {

constexpr int CT_UNROLL = 4;
constexpr int CT_THREADS = 128;          // block of k_count_tab: four warps, or one group
constexpr int CT_WORDS = 4096;           // its table: a quarter per warp, or the whole
constexpr int CT_FILL_WARP = CT_WORDS / (CT_THREADS / 32) * 3 / 4;
constexpr int CT_BLOCKS = 8;             // resident blocks per SM
constexpr int CT_FILL_GROUP = CT_WORDS * 3 / 4;
constexpr int CT_LATE = 32 * (CT_UNROLL + 1);  // waiting entries of a warp at most
constexpr int CB_THREADS = 512;          // block of k_count_big, two per SM
constexpr int CB_WORDS = 8192;
constexpr int CB_FILL = CB_WORDS * 3 / 4;
constexpr int CB_WORDS_LONG = 16384;     // the table of its unstaged runs
constexpr int CB_FILL_LONG = CB_WORDS_LONG * 3 / 4;
constexpr int CB_STAGE = CB_FILL + 8;    // entries of a staging buffer (a run may start mid 16 bytes)
// Label ids below this take the one-word tables: at least 12 bits are then left
// for the repeats, so that runs of up to 4095 entries (8191 below 2^19 ids, any
// run of the classes above below 2^18) fit; with more ids too many runs would
// fall to the hash classes.
constexpr int CT_MAX_K = 1 << 20;

// Bits of a word left for the repeats when every key + 1 is at most K.
__host__ __device__ inline int ct_count_bits(int K)
{
    int kb = 1;
    while (kb < 31 && (1u << kb) <= (unsigned)K) ++kb;
    return 32 - kb;
}

// Slots of a run of m entries: the power of two of at least 4/3 m (and 32).
__device__ __forceinline__ unsigned ct_slots_log2(unsigned m)
{
    const unsigned need = (4u * m + 2u) / 3u;
    return need <= 32u ? 5u : 32u - (unsigned)__clz((int)(need - 1u));
}

// Barrier of a group: a warp, or the whole block (its size known at compile
// time: a barrier number computed at run time would reserve all sixteen of a
// block's hardware barriers and so limit the resident blocks to four).
template <int GS>
__device__ __forceinline__ void ct_sync()
{
    if (GS == 32) __syncwarp();
    else block_sync();
}

// Warp total of a pair sum below 2^162 (valid in every lane): six 27-bit
// chunks, whose sums over 32 lanes fit 32 bits, each added by one redux
// instead of five rounds of shuffles and carries.
__device__ __forceinline__ U192 ct_warp_sum(const U192 &a)
{
    constexpr unsigned M = (1u << 27) - 1u, ALL = 0xffffffffu;
    const unsigned w0 = (unsigned)a.w0, w1 = (unsigned)(a.w0 >> 32), w2 = (unsigned)a.w1, w3 = (unsigned)(a.w1 >> 32),
                   w4 = (unsigned)a.w2, w5 = (unsigned)(a.w2 >> 32);
    const unsigned c[6] = {w0 & M, __funnelshift_r(w0, w1, 27) & M, __funnelshift_r(w1, w2, 22) & M,
                           __funnelshift_r(w2, w3, 17) & M, __funnelshift_r(w3, w4, 12) & M,
                           __funnelshift_r(w4, w5, 7) & M};
    unsigned s[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) s[k] = __reduce_add_sync(ALL, c[k]);
    U192 r;
    const u128 lo = (u128)s[0] + ((u128)s[1] << 27) + ((u128)s[2] << 54);    // below 2^87
    const u128 hi = (u128)s[3] + ((u128)s[4] << 27) + ((u128)s[5] << 54);    // times 2^81, below 2^87
    const u128 hs = hi << 17;                                                // times 2^64, below 2^104
    r.w0 = (unsigned long long)lo;
    const u128 t = (lo >> 64) + hs;
    r.w1 = (unsigned long long)t;
    r.w2 = (unsigned long long)(t >> 64);
    return r;
}

// Group totals of the counts (below 2^32) and pair sums, for the group's
// first thread (8 words per warp in red).
template <bool FULL, int GS>
__device__ __forceinline__ void ct_totals(unsigned (&counts)[3], U192 &inner, U192 &inner_full, unsigned long long *red)
{
#pragma unroll
    for (int k = 0; k < 3; ++k) counts[k] = __reduce_add_sync(0xffffffffu, counts[k]);
    inner = ct_warp_sum(inner);
    if (FULL) inner_full = ct_warp_sum(inner_full);
    if (GS == 32) return;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) {
        unsigned long long *r = red + 8 * wid;
        r[0] = ((unsigned long long)counts[2] << 32) | counts[0];
        r[1] = counts[1];
        r[2] = inner.w0;
        r[3] = inner.w1;
        r[4] = inner.w2;
        if (FULL) {
            r[5] = inner_full.w0;
            r[6] = inner_full.w1;
            r[7] = inner_full.w2;
        }
    }
    ct_sync<GS>();
    if (threadIdx.x == 0)
        for (int w = 1; w < GS / 32; ++w) {
            const unsigned long long *r = red + 8 * w;
            counts[0] += (unsigned)r[0];
            counts[2] += (unsigned)(r[0] >> 32);
            counts[1] += (unsigned)r[1];
            u192_add(inner, U192{r[2], r[3], r[4]});
            if (FULL) u192_add(inner_full, U192{r[5], r[6], r[7]});
        }
}

// a += r, as one carry chain.
__device__ __forceinline__ void u192_add_chain(U192 &a, const Rcp &r)
{
    asm("add.cc.u64 %0, %0, %3;\n\taddc.cc.u64 %1, %1, %4;\n\taddc.u64 %2, %2, 0;"
        : "+l"(a.w0), "+l"(a.w1), "+l"(a.w2)
        : "l"(r.lo), "l"(r.hi));
}

// Follows up to 32 entries whose first slot was taken (one per lane, key = 0
// for none) to their key's slot or a free one.  Returns the occurrences of the
// key before this one.
__device__ __forceinline__ unsigned ct_follow(unsigned *slot, unsigned key, unsigned mask, unsigned shift, int cb)
{
    unsigned before = 0u, h = ((key - 1u) * 0x9E3779B1u) >> shift;
    bool pend = key != 0u;
    // bounded: the slots of a run are never all taken
    for (unsigned step = 0; step <= mask && __any_sync(0xffffffffu, pend); ++step) {
        if (pend) {
            const unsigned cur = atomicCAS(&slot[h], 0u, key << cb);
            const bool own = (cur >> cb) == key;
            if (own) before = (atomicAdd(&slot[h], 1u) & ((1u << cb) - 1u)) + 1u;
            pend = cur != 0u && !own;
            h = (h + 1u) & mask;
        }
    }
    __syncwarp();
    return before;
}

// What the runs hold: every label != c, of which only those above c are
// counted here (CT_MIXED: each unordered pair is charged to its smaller id), or
// only labels above c (CT_ABOVE); or every label != c with c's own penalty S_c
// formed beside T_c (CT_FULL).
enum { CT_MIXED = 0, CT_ABOVE = 1, CT_FULL = 2 };

// Counts the m entries of run h (labels at src, in shared or global memory)
// with a group of GS threads and writes community h.c's record.  slot holds
// at least 2^ct_slots_log2(m) zero words and is left zero; late is the warp's
// CT_LATE words.  The steps are warp-uniform, so that the warp issues each
// once for all lanes; only the last step of a run checks its bounds.
template <int MODE, bool SMEM, int GS>
__device__ __forceinline__ void ct_count_run(const CountCtx &x, const RunHdr &h, const int *src, unsigned *slot, int cb,
                                             int gtid, unsigned *late, unsigned long long *red)
{
    constexpr unsigned ALL = 0xffffffffu;
    constexpr bool FULL = MODE == CT_FULL;
    const int m = (int)h.m, c = h.c, lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u, one = 1u << cb;
    const unsigned lg = ct_slots_log2(h.m), mask = (1u << lg) - 1u, shift = 32u - lg;
    // the repeats; twice the occurrences before each, summed (with the entries:
    // the sum of the squares); the entries counted (CT_ABOVE: all m)
    unsigned counts[3] = {0u, 0u, 0u};
    unsigned nl = 0;  // entries waiting in `late`
    U192 inner, inner_full;
    u192_zero(inner);
    u192_zero(inner_full);
    auto follow = [&](unsigned n) {  // the last n <= 32 waiting entries
        nl -= n;
        const unsigned key = (unsigned)lane < n ? late[nl + lane] : 0u;
        const unsigned before = ct_follow(slot, key, mask, shift, cb);
        if (__any_sync(ALL, before != 0u)) {
            if (before) {
                const Rcp r = ld_rcp(&x.recip[key - 1u]);
                if (FULL) u192_mac(inner_full, 2u * before, r);
                if (!FULL || (int)(key - 1u) > c) {
                    u192_mac(inner, 2u * before, r);
                    counts[0] += 1u;
                    counts[1] += 2u * before;
                }
            }
            __syncwarp();
        }
    };
    auto label = [&](int e) { return SMEM ? src[e] : __ldcs(&src[e]); };
    int nx[CT_UNROLL];
#pragma unroll
    for (int k = 0; k < CT_UNROLL; ++k) nx[k] = label(max(0, min(gtid + GS * k, m - 1)));  // (an empty run reads the slack)
    // one step of CT_UNROLL entries a lane from e0 (warp-uniform) on
    auto step = [&](int e0, auto last) {
        constexpr bool LAST = decltype(last)::value;
        constexpr bool EVERY = !LAST && MODE != CT_MIXED && !QM_CHECKED;  // no entry is skipped
        int lv[CT_UNROLL];
        unsigned cur[CT_UNROLL];
        Rcp rj[CT_UNROLL];
#pragma unroll
        for (int k = 0; k < CT_UNROLL; ++k) {
            lv[k] = nx[k];
            if ((LAST && e0 + lane + GS * k >= m) || (MODE == CT_MIXED && lv[k] < c) || !QM_CHK(lv[k], x.K, 6))
                lv[k] = -1;
            if (!EVERY) rj[k] = Rcp{0ull, 0ull};
            if (EVERY || lv[k] >= 0) rj[k] = ld_rcp(&x.recip[lv[k]]);
        }
        if (!LAST)
#pragma unroll
            for (int k = 0; k < CT_UNROLL; ++k)  // the next step's labels
                nx[k] = label(min(e0 + lane + GS * (CT_UNROLL + k), m - 1));
#pragma unroll
        for (int k = 0; k < CT_UNROLL; ++k) {
            const unsigned hs = ((unsigned)lv[k] * 0x9E3779B1u) >> shift;
            cur[k] = 0u;
            if (EVERY || lv[k] >= 0) cur[k] = atomicCAS(&slot[hs], 0u, (unsigned)lv[k] * one + one);
        }
#pragma unroll
        for (int k = 0; k < CT_UNROLL; ++k) {
            const unsigned taken = __ballot_sync(ALL, cur[k] != 0u);
            if (cur[k] != 0u) late[nl + __popc(taken & lt)] = (unsigned)lv[k] + 1u;
            nl += __popc(taken);
        }
        __syncwarp();
        while (nl >= 32u) follow(32u);
#pragma unroll
        for (int k = 0; k < CT_UNROLL; ++k) {
            if (FULL) {
                u192_add_chain(inner_full, rj[k]);
                const bool above = lv[k] > c;  // else the pair is charged to the other community
                rj[k].lo = above ? rj[k].lo : 0ull;
                rj[k].hi = above ? rj[k].hi : 0ull;
                counts[2] += above ? 1u : 0u;
            } else if (MODE == CT_MIXED || QM_CHECKED) {
                counts[2] += lv[k] >= 0 ? 1u : 0u;
            }
            u192_add_chain(inner, rj[k]);
        }
    };
    int e0 = gtid & ~31;
    for (; e0 + GS * (CT_UNROLL - 1) + 32 <= m; e0 += GS * CT_UNROLL) step(e0, std::false_type{});
    if (e0 < m) step(e0, std::true_type{});
    if (nl) follow(nl);
    ct_sync<GS>();
    for (unsigned i = (unsigned)gtid; i < (1u << lg) / 4u; i += (unsigned)GS)
        reinterpret_cast<uint4 *>(slot)[i] = make_uint4(0u, 0u, 0u, 0u);
    ct_totals<FULL, GS>(counts, inner, inner_full, red);
    if (gtid == 0) {
        const unsigned long long entries = MODE == CT_ABOVE && !QM_CHECKED ? (unsigned)m : counts[2];
        put_record(x, c, h.vol, h.m, entries - counts[0], entries + counts[1], inner, inner_full);
    }
    ct_sync<GS>();  // the cleared slots and `red` are free for the next run
}

}  // namespace qmk
