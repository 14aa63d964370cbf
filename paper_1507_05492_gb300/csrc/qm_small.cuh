// qm_small.cuh -- a comparison of two small labellings in one kernel (included by
// qm_kernels.cu).
//
// On a few thousand nodes the comparison's nine kernels are a chain of launches
// that wait on one another; the work itself is some microseconds, most of it
// FP64, which an SM issues at two operations a cycle.  So one cluster of eight
// blocks does it all: every block reads all labels and keeps the found
// communities b with b mod 8 equal to its rank, whose cells it counts in a
// shared-memory table; the truth sizes and row maxima are shared through global
// memory, with a cluster barrier between the phases; and the result is written
// straight to the caller's pinned memory.  The terms are the other path's
// functions and every sum is exact, so the results are the same bits.
// 10^4 nodes: 109 -> 54 us a call (bound by its chains of dependent FP64
// operations: a division, a logarithm and a barrier after another); beyond CS_MAX_NODES a block's shared memory may not hold its cells.
// Included inside namespace qm of qm_kernels.cu, after the helpers it uses.

constexpr int CS_CTAS = 8, CS_THREADS = 512;
constexpr int CS_MAX_SLOTS = 21504;  // 10 bytes each: a block may come to hold every cell
constexpr int CS_MAX_NODES = CS_MAX_SLOTS * 3 / 4;
constexpr int CS_MAX_K = 1 << 16;
// Beyond this many nodes two labellings that both have communities of fewer than
// 8/3 nodes on average go the other path.  Communities of two on both sides, this
// path and the other, us: 10^4 nodes 103 and 108, 12,000 114 and 109, 16,128 141 and
// 120 (of three, 16,128 nodes: 91 and 108; of two against 30 79 and 114).
constexpr int CS_FINE_NODES = 10000;

struct CompareSmallArgs {
    const int *truth, *found;
    int n, ka, kb, abits, slots;
    int *size_a, *size_b;            // [ka], [kb]
    unsigned *rowmax_n, *colmax;     // [ka], [kb]
    unsigned long long *rowmax_r;    // [ka]
    unsigned long long *g;           // GC_* words
    int *status;
    qm_compare *out;                 // pinned host memory
    int *out_status;
};

__global__ void __cluster_dims__(CS_CTAS, 1, 1) __launch_bounds__(CS_THREADS) k_compare_small(CompareSmallArgs a)
{
    extern __shared__ __align__(16) unsigned sm_small[];
    __shared__ int s_cells;
    __shared__ __align__(8) unsigned wait_s[CS_THREADS / 32][64];
    __shared__ unsigned late_s[CS_THREADS / 32][LATE_CELL_WORDS];
    __shared__ double s_ones[2];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, rank = blockIdx.x;
    const int gt = rank * CS_THREADS + tid, GT = CS_CTAS * CS_THREADS;
    unsigned *const key = sm_small, *const cnt = sm_small + a.slots;
    unsigned short *const list = (unsigned short *)(cnt + a.slots);  // the slots taken
    if (tid == 0) s_cells = 0;
    for (int i = tid; i < a.slots / 2; i += CS_THREADS)
        reinterpret_cast<uint4 *>(sm_small)[i] = make_uint4(0u, 0u, 0u, 0u);
    for (int i = gt; i < a.ka; i += GT) {
        a.size_a[i] = 0;
        a.rowmax_n[i] = 0u;
        a.rowmax_r[i] = 0ull;
    }
    for (int i = gt; i < a.kb; i += GT) {
        a.size_b[i] = 0;
        a.colmax[i] = 0u;
    }
    if (gt < GC_COUNT) a.g[gt] = 0ull;
    if (gt == GC_COUNT) *a.status = 0;
    if (tid == CS_THREADS - 1) {
        s_ones[0] = nmi_over(1, a.n);
        s_ones[1] = log_ratio(a.n, 1);
    }
    cluster_sync();

    // cells of this block's found communities
    unsigned *const wait = wait_s[wid];
    unsigned nl = 0;
    bool bad = false;
    auto follow = [&](unsigned m) {  // the last m <= 32 keys whose first slot was another's
        nl -= m;
        const unsigned k = (unsigned)lane < m ? wait[nl + lane] : 0u;
        unsigned h = tab_hash(k, a.slots);
        bool pend = k != 0u;
        // bounded: at most 3/4 of the slots are ever taken
        for (int step = 0; step < a.slots && __any_sync(0xffffffffu, pend); ++step) {
            if (pend) {
                h = h + 1u == (unsigned)a.slots ? 0u : h + 1u;
                const unsigned v = atomicCAS(&key[h], 0u, k);
                if (v == 0u || v == k) {
                    atomicAdd(&cnt[h], 1u);
                    pend = false;
                }
            }
        }
        __syncwarp();
    };
    for (int i0 = tid & ~31; i0 < a.n; i0 += 4 * CS_THREADS) {
        int x[4], b[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = i0 + lane + q * CS_THREADS;
            x[q] = i < a.n ? __ldg(&a.truth[i]) : -2;
            b[q] = i < a.n ? __ldg(&a.found[i]) : -2;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const bool ok = (unsigned)x[q] < (unsigned)a.ka && (unsigned)b[q] < (unsigned)a.kb;
            if (!ok && i0 + lane + q * CS_THREADS < a.n) bad = true;
            const unsigned k = ok && (b[q] & (CS_CTAS - 1)) == rank ? (((unsigned)b[q] << a.abits) | (unsigned)x[q]) + 1u : 0u;
            const unsigned h = tab_hash(k, a.slots);
            unsigned v = k;
            if (k) {
                v = atomicCAS(&key[h], 0u, k);
                if (v == 0u) v = k;
                if (v == k) atomicAdd(&cnt[h], 1u);
            }
            const unsigned mm = __ballot_sync(0xffffffffu, v != k);
            if (v != k) wait[nl + __popc(mm & ((1u << lane) - 1u))] = k;
            nl += (unsigned)__popc(mm);
            __syncwarp();
            if (nl >= 32u) follow(32u);
        }
    }
    if (nl) follow(nl);
    if (bad) atomicOr(a.status, 1);
    block_sync();

    // sizes of both sides and column maxima
    const unsigned amask = (1u << a.abits) - 1u;
    CompareAcc acc;
    compare_acc_zero(acc);
    for (int i0 = tid & ~31; i0 < a.slots; i0 += CS_THREADS) {
        const int i = i0 + lane;
        const unsigned v = i < a.slots ? key[i] : 0u;
        const unsigned m = __ballot_sync(0xffffffffu, v != 0u);
        if (!m) continue;
        int at = 0;
        if (lane == 0) at = atomicAdd(&s_cells, __popc(m));
        at = __shfl_sync(0xffffffffu, at, 0);
        if (v) {
            list[at + __popc(m & ((1u << lane) - 1u))] = (unsigned short)i;
            const unsigned n = cnt[i];
            const int x = (int)((v - 1u) & amask), b = (int)((v - 1u) >> a.abits);
            atomicAdd(&a.size_a[x], (int)n);
            atomicAdd(&a.size_b[b], (int)n);
            atomicMax(&a.colmax[b], n);
            acc.cells += 1;
        }
        __syncwarp();
    }
    cluster_sync();
    if (__ldcg(a.status)) {  // a label out of range
        if (gt == 0) {
            *a.out_status = __ldcg(a.status);
            __threadfence_system();
        }
        return;
    }

    // terms of the cells and of this block's columns
    LateCells lc{late_s[wid], true, s_ones[0], s_ones[1]};
    const int ncells = s_cells;
    for (int i0 = tid & ~31; i0 < ncells; i0 += CS_THREADS) {
        const bool in = i0 + lane < ncells;
        const int i = in ? list[i0 + lane] : 0;
        const unsigned v = in ? key[i] : 0u;
        unsigned n = 0, na = 0, nb = 0;
        if (in) {
            n = cnt[i];
            const int x = (int)((v - 1u) & amask), b = (int)((v - 1u) >> a.abits);
            na = (unsigned)__ldcg(&a.size_a[x]);
            nb = (unsigned)__ldcg(&a.size_b[b]);
            acc.a11 += (unsigned long long)n * (n - 1u) / 2ull;
            atomicMax(&a.rowmax_n[x], n);
            rowmax_ratio_update(&a.rowmax_r[x], n, (unsigned long long)na + nb);
        }
        cell_terms_warp(n, na, nb, in, a.n, nullptr, acc, lc);
    }
    late_cells_flush_block(late_s[0], wait_s[0], a.n, nullptr, acc, lc);
    // (from the block's last thread on: its first warps are at the waiting cells)
    for (int b = rank + CS_CTAS * (CS_THREADS - 1 - tid); b < a.kb; b += CS_CTAS * CS_THREADS) {
        const long long nb = __ldcg(&a.size_b[b]);
        if (nb == 0) continue;
        acc.sb += (unsigned long long)(nb * (nb - 1) / 2);
        acc.nvd += __ldcg(&a.colmax[b]);
        acc.hden += fp_from_double(entropy_term(nb, a.n), SC_H);
        acc.kb += 1;
    }
    cluster_sync();

    // rows
    for (int x = rank + CS_CTAS * tid; x < a.ka; x += CS_CTAS * CS_THREADS) {
        const long long na = __ldcg(&a.size_a[x]);
        if (na == 0) continue;
        const unsigned long long f = __ldcg(&a.rowmax_r[x]);
        const long long fn = (long long)(f >> 32), fd = (long long)(f & 0xFFFFFFFFull);
        acc.sa += (unsigned long long)(na * (na - 1) / 2);
        acc.nvd += __ldcg(&a.rowmax_n[x]);
        acc.f += fp_from_double(__dmul_rn((double)na, f_ratio(fn, na, fd - na)), SC_F);
        acc.hden += fp_from_double(entropy_term(na, a.n), SC_H);
        acc.ka += 1;
    }
    __syncwarp();
    static_assert(2 * GC_COUNT <= 64, "a warp's words take the place of its waiting keys");
    unsigned long long *const words = (unsigned long long *)wait_s[wid];
    compare_words_warp(acc, words);
    block_sync();
    if (tid < GC_COUNT) {
        unsigned long long t = 0;
        for (int w = 0; w < CS_THREADS / 32; ++w) t += ((const unsigned long long *)wait_s[w])[tid];
        if (t) atomicAdd(a.g + tid, t);
    }
    cluster_sync();
    if (rank == 0 && wid == 0) {
        if (lane < GC_COUNT) words[lane] = __ldcg(&a.g[lane]);
        __syncwarp();
        compare_warp(words, a.n, a.out);
        __threadfence_system();
        __syncwarp();
    }
    if (gt == 0) {
        *a.out_status = 0;
        __threadfence_system();
    }
}
