// qm_cells.cuh -- contingency cells of two large labellings by buckets of found
// communities (included by qm_kernels.cu).
//
// Every index with ground truth comes from the cells |c n c'|.  On large inputs
// the counting sort of the nodes by found label writes 4 bytes a node at random
// over an array larger than L2, and its histogram is an atomic a node.  Here the
// nodes are split instead by ranges of found labels ("buckets") in two passes
// with sequential traffic, and each bucket's cells are counted in shared memory:
//   k_cells_count  nodes of every (bucket, tile of CELL_TILE nodes);
//   (a scan gives every group's place, bucket by bucket)
//   k_cells_split  per tile: (truth, found) pairs into shared memory grouped by
//                  bucket, then every group to its place, 4 bytes a node;
//   k_cells_table  per bucket: a hash table of its cells; the cells go out in
//                  one stretch, the sizes of both sides are summed from them.
// The cells are the same multiset as the counting sort's, and every sum over
// them is exact, so the results are the same bits.
//
// Measured at 10^8 nodes against the sort (k_hist, k_scatter, k_compare_cm):
// 4.15 -> 1.38 ms with 20% of the nodes moved (count 0.11, scan 0.06, split
// 0.48, table 0.73; the split is bound by its short groups, the table by
// shared-memory atomics), 1.18 with 1% moved, 1.85 with half moved.  2^13
// buckets with two smaller tables an SM: split 0.65, table 0.79 ms; 2^12 with
// tables of 11,264 slots, which half moved labels overflow: table 0.93 and 3.76
// ms.  At 3*10^6 nodes the whole call takes 0.22 ms.
// Included inside namespace qm of qm_kernels.cu, after the helpers it uses.

constexpr int CELL_BITS = 12;                  // at most 2^12 buckets
constexpr int CELL_BUCKET = 24576;             // nodes of a bucket aimed at: their cells mostly fit the table
constexpr int CELL_THREADS = 1024;             // the passes over tiles
constexpr int CELL_TILE = 45056;               // nodes of a tile: 4 bytes each beside two words a bucket
constexpr int CELL_TAB_THREADS = 1024;
constexpr int CELL_SLOTS = 24576;              // slots of a bucket's table (8 bytes each), one block per SM
constexpr int CELL_FILL = CELL_SLOTS * 3 / 4;
constexpr int CELL_MAX_RANGE = 1024;           // found labels of a bucket
// (A tile a third of the SMs.  20% moved, sort and buckets, us a call: 2.2*10^6 nodes
// 252 and 152, 3*10^6 316 and 183.)
constexpr long long CELL_MIN_NODES = 1LL << 21;

struct CellPlan {
    int sh;      // bucket of a found label b: b >> sh
    int nb;      // buckets
    int ntiles;
    bool ok;
};

static int bits_of(long long k)  // bits that hold 0 .. k - 1
{
    int b = 0;
    while ((1LL << b) < k) ++b;
    return b;
}

// Whether the buckets apply: enough nodes to fill the GPU with tiles, and a
// truth label with a bucket's part of a found label in 32 bits (one value kept
// for "no entry").
static CellPlan cell_plan(long long n, int ka, int kb)
{
    CellPlan p;
    const int bits = std::min(CELL_BITS, std::max(8, bits_of((n + CELL_BUCKET - 1) / CELL_BUCKET)));
    p.sh = std::max(0, bits_of(kb) - bits);
    p.nb = (int)(((long long)kb + (1LL << p.sh) - 1) >> p.sh);
    p.ntiles = (int)((n + CELL_TILE - 1) / CELL_TILE);
    p.ok = n > CELL_MIN_NODES && (1LL << p.sh) <= CELL_MAX_RANGE && bits_of(ka) + p.sh <= 31 &&
           (long long)p.nb * p.ntiles < (1LL << 30);
    return p;
}

struct CellArgs {
    const int *truth, *found;
    long long n;
    int ka, kb, sh, nb, ntiles;
    int *off;            // [nb * ntiles + 1] counts, then places (bucket-major)
    unsigned *pairs;     // [n] (found low bits << abits | truth), by bucket
    int abits;
    Cell *cells;
    int *ncells;
    int *size_a, *size_b;
    unsigned long long *gacc;
    int *next;           // claim counter of k_cells_table
    int *status;
};

__global__ void __launch_bounds__(CELL_THREADS) k_cells_count(CellArgs a)
{
    __shared__ int cnt[1 << CELL_BITS];
    bool bad = false;
    for (int t = blockIdx.x; t < a.ntiles; t += gridDim.x) {
        for (int i = threadIdx.x; i < a.nb; i += CELL_THREADS) cnt[i] = 0;
        __syncthreads();
        const long long u0 = (long long)t * CELL_TILE, u1 = min(a.n, u0 + CELL_TILE);
        for (long long i0 = u0 + threadIdx.x; i0 < u1; i0 += 4 * CELL_THREADS) {
            int b[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const long long i = i0 + k * CELL_THREADS;
                b[k] = i < u1 ? __ldcs(&a.found[i]) : -2;
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if ((unsigned)b[k] < (unsigned)a.kb) atomicAdd(&cnt[b[k] >> a.sh], 1);
                else if (i0 + k * CELL_THREADS < u1) bad = true;
            }
        }
        __syncthreads();
        for (int i = threadIdx.x; i < a.nb; i += CELL_THREADS) a.off[(long long)i * a.ntiles + t] = cnt[i];
        __syncthreads();
    }
    if (bad) atomicOr(a.status, 1);
}

constexpr int CELL_SPLIT_SMEM = CELL_TILE * 4 + 2 * (1 << CELL_BITS) * 4;

__global__ void __launch_bounds__(CELL_THREADS) k_cells_split(CellArgs a)
{
    extern __shared__ __align__(16) unsigned sm_cells[];
    __shared__ unsigned long long red[72];
    if (block_stopped(a.status)) return;
    unsigned *const buf = sm_cells;                    // the tile's pairs, by bucket
    int *const cur = (int *)(buf + CELL_TILE);         // local cursors; at the end each group's end
    int *const go = cur + (1 << CELL_BITS);            // global place of each group
    constexpr int PER = (1 << CELL_BITS) / CELL_THREADS;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const unsigned low = (1u << a.sh) - 1u;
    bool bad = false;
    for (int t = blockIdx.x; t < a.ntiles; t += gridDim.x) {
        int c[PER];
        unsigned sum = 0;
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            const int b = tid * PER + k;
            c[k] = 0;
            if (b < a.nb) {
                const long long i = (long long)b * a.ntiles + t;
                const int o = a.off[i];
                go[b] = o;
                c[k] = a.off[i + 1] - o;
            }
            sum += (unsigned)c[k];
        }
        unsigned excl;
        group_exclusive_scan(sum, excl, CELL_THREADS, red);
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            cur[tid * PER + k] = (int)excl;
            excl += (unsigned)c[k];
        }
        __syncthreads();
        const long long u0 = (long long)t * CELL_TILE, u1 = min(a.n, u0 + CELL_TILE);
        for (long long i0 = u0 + tid; i0 < u1; i0 += 4 * CELL_THREADS) {
            int x[4], b[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const long long i = i0 + k * CELL_THREADS;
                x[k] = i < u1 ? __ldcs(&a.truth[i]) : 0;
                b[k] = i < u1 ? __ldcs(&a.found[i]) : -1;
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (b[k] < 0) continue;
                if ((unsigned)x[k] >= (unsigned)a.ka) {
                    bad = true;
                    x[k] = 0;
                }
                buf[atomicAdd(&cur[b[k] >> a.sh], 1)] = (((unsigned)b[k] & low) << a.abits) | (unsigned)x[k];
            }
        }
        __syncthreads();
        // every group to its place, a half-warp per group (a dozen pairs at 4096 buckets)
        const int hw = (wid << 1) | (lane >> 4), hl = lane & 15;
        for (int b = hw; b < a.nb; b += 2 * (CELL_THREADS / 32)) {
            const int s = b ? cur[b - 1] : 0, e = cur[b], o = go[b] - s;
            for (int k = s + hl; k < e; k += 16) a.pairs[o + k] = buf[k];
        }
        __syncthreads();
    }
    if (bad) atomicOr(a.status, 1);
}

constexpr int CELL_TAB_SMEM = CELL_SLOTS * 8;

// Cells of the buckets, a block each (claimed in turn).  A slot is a key word
// ((found low bits << abits | truth) + 1, 0 free) and a count word; a bucket with
// more cells than the table takes is split into hash classes, each of which is
// emitted when it fits.
__global__ void __launch_bounds__(CELL_TAB_THREADS, 1) k_cells_table(CellArgs a)
{
    extern __shared__ __align__(16) unsigned sm_tab[];
    __shared__ int nbs[CELL_MAX_RANGE];
    __shared__ unsigned colmax[CELL_MAX_RANGE];
    __shared__ unsigned long long red[72];
    __shared__ unsigned late_s[CELL_TAB_THREADS / 32][32 * 5];
    __shared__ int s_b, s_used, s_at, s_over;
    __shared__ unsigned s_done;
    if (block_stopped(a.status)) return;
    unsigned *const key = sm_tab, *const cnt = sm_tab + CELL_SLOTS;
    const int tid = threadIdx.x, lane = tid & 31;
    const int range = 1 << a.sh;
    const unsigned amask = (1u << a.abits) - 1u;
    unsigned long long nvd = 0, ncell = 0;
    unsigned *const late = late_s[tid >> 5];
    unsigned nl = 0;
    // follows the last n <= 32 waiting keys to their slots; returns the new ones.
    // Bounded: keys stop being added at 3/4 of the slots, and a warp adds at most
    // 5 * 32 after that, so a free slot remains.
    auto follow = [&](unsigned n) {
        nl -= n;
        const unsigned k = (unsigned)lane < n ? late[nl + lane] : 0u;
        unsigned h = tab_hash(k, CELL_SLOTS);
        bool pend = k != 0u, take = false;
        for (int step = 0; step < CELL_SLOTS && __any_sync(0xffffffffu, pend); ++step) {
            if (pend) {
                h = h + 1u == (unsigned)CELL_SLOTS ? 0u : h + 1u;
                unsigned v = ((volatile unsigned *)key)[h];
                if (v == 0u) {
                    v = atomicCAS(&key[h], 0u, k);
                    take = v == 0u;
                    if (take) v = k;
                }
                if (v == k) atomicAdd(&cnt[h], 1u);
                pend = v != k;
            }
        }
        __syncwarp();
        return (unsigned)__popc(__ballot_sync(0xffffffffu, take));
    };
    for (int i = tid; i < CELL_SLOTS / 2; i += CELL_TAB_THREADS)
        reinterpret_cast<uint4 *>(sm_tab)[i] = make_uint4(0u, 0u, 0u, 0u);
    for (;;) {
        if (tid == 0) s_b = atomicAdd(a.next, 1);
        for (int i = tid; i < range; i += CELL_TAB_THREADS) {
            nbs[i] = 0;
            colmax[i] = 0u;
        }
        if (tid == 0) {
            s_used = s_over = 0;
            s_done = 0u;
        }
        block_sync();
        const int bk = s_b;
        if (bk >= a.nb) break;
        // (unsigned: the steps of the walk pass 2^31 in the last bucket of that many nodes)
        const unsigned p0 = a.off[(long long)bk * a.ntiles], p1 = a.off[(long long)(bk + 1) * a.ntiles];
        // classes still to do: hash class r of R, split in two when it overflows
        // (the second halves wait as bits of `todo`, one per doubling)
        unsigned r = 0, R = 1;
        unsigned long long todo = 0;
        while (p0 < p1) {
            for (unsigned i0 = p0 + (tid & ~31); i0 < p1; i0 += 4 * CELL_TAB_THREADS) {
                unsigned k[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const unsigned i = i0 + lane + q * CELL_TAB_THREADS;
                    k[q] = i < p1 ? __ldcs(&a.pairs[i]) + 1u : 0u;
                    if (R > 1 && tab_split(k[q], R) != r) k[q] = 0u;
                }
                // more keys than the table takes; or, once it is half as full, so many per entry
                // that the rest would bring them (found at the end, a nearly full table of long
                // probes would have been filled for nothing: 10^8 nodes, two labellings at
                // random, this kernel 7.7 and 3.0 ms; 10^7 nodes 1.04 and 0.42)
                const int have = *(volatile int *)&s_used;
                const unsigned read = *(volatile unsigned *)&s_done;
                if (have > CELL_FILL ||
                    (have > CELL_FILL / 2 && (long long)have * (p1 - p0) > (long long)CELL_FILL * read))
                    *(volatile int *)&s_over = 1;
                if (__any_sync(0xffffffffu, *(volatile int *)&s_over)) break;  // this class does not fit: stop reading it
                // first slots of all four: own key or free; the others are followed 32 at a time
                unsigned fresh = 0;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const unsigned h = tab_hash(k[q], CELL_SLOTS);
                    unsigned v = k[q] ? ((volatile unsigned *)key)[h] : 0u;
                    bool take = false;
                    if (k[q] && v == 0u) {
                        v = atomicCAS(&key[h], 0u, k[q]);
                        take = v == 0u;
                        if (take) v = k[q];
                    }
                    if (k[q] && v == k[q]) atomicAdd(&cnt[h], 1u);
                    const bool miss = v != k[q];
                    fresh += (unsigned)__popc(__ballot_sync(0xffffffffu, take));
                    const unsigned mm = __ballot_sync(0xffffffffu, miss);
                    if (miss) late[nl + __popc(mm & ((1u << lane) - 1u))] = k[q];
                    nl += (unsigned)__popc(mm);
                }
                __syncwarp();
                while (nl >= 32u) fresh += follow(32u);
                if (lane == 0) {
                    atomicAdd(&s_done, 128u);
                    if (fresh) atomicAdd(&s_used, (int)fresh);
                }
            }
            {
                // (other warps may be setting the flag: one answer for the warp, which follow() needs whole)
                const bool over = __any_sync(0xffffffffu, *(volatile int *)&s_over);
                const unsigned fresh = nl && !over ? follow(nl) : 0u;
                nl = 0;
                if (lane == 0 && fresh) atomicAdd(&s_used, (int)fresh);
            }
            block_sync();
            const int used = s_used;
            const bool split = s_over != 0 || used > CELL_FILL;
            if (split) {  // nothing is emitted: the class is split in two
                for (int i = tid; i < CELL_SLOTS / 2; i += CELL_TAB_THREADS)
                    reinterpret_cast<uint4 *>(sm_tab)[i] = make_uint4(0u, 0u, 0u, 0u);
                if (R >= (1u << 30)) {
                    if (tid == 0) atomicOr(a.status, 2);
                    block_sync();
                    break;
                }
                todo |= (unsigned long long)R;  // class (r + R) of 2R waits
                R *= 2u;
            } else {
                if (tid == 0) s_at = atomicAdd(a.ncells, used);
                block_sync();
                for (int i0 = tid & ~31; i0 < CELL_SLOTS; i0 += CELL_TAB_THREADS) {
                    const int i = i0 + lane;
                    const unsigned v = key[i];
                    const unsigned m = __ballot_sync(0xffffffffu, v != 0u);
                    if (!m) continue;
                    int at = 0;
                    if (lane == 0) at = atomicAdd(&s_at, __popc(m));
                    at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & ((1u << lane) - 1u));
                    if (v) {
                        const unsigned n = cnt[i];
                        const int x = (int)((v - 1u) & amask), lo = (int)((v - 1u) >> a.abits);
                        a.cells[at] = Cell{x, (bk << a.sh) + lo, n, 0u};
                        atomicAdd(&a.size_a[x], (int)n);
                        atomicAdd(&nbs[lo], (int)n);
                        atomicMax(&colmax[lo], n);
                        key[i] = 0u;
                        cnt[i] = 0u;
                    }
                    __syncwarp();
                }
                if (tid == 0) ncell += (unsigned long long)used;
                // the next class: the second half of the deepest split still waiting
                if (!todo) {
                    block_sync();
                    break;
                }
                const unsigned top = 1u << (63 - __clzll((long long)todo));
                todo &= ~(unsigned long long)top;
                r = (r & (top - 1u)) + top;
                R = 2u * top;
            }
            block_sync();
            if (tid == 0) {
                s_used = s_over = 0;
                s_done = 0u;
            }
            block_sync();
        }
        block_sync();
        for (int i = tid; i < range; i += CELL_TAB_THREADS) {
            const long long b = ((long long)bk << a.sh) + i;
            if (b < a.kb) a.size_b[b] = nbs[i];
            nvd += colmax[i];
        }
        block_sync();
    }
    const unsigned long long t = group_sum_u64(nvd, CELL_TAB_THREADS, red);
    if (tid == 0) {
        if (t) atomicAdd(a.gacc + GC_NVD, t);
        if (ncell) atomicAdd(a.gacc + GC_CELLS, ncell);
    }
}
