// qm_reorder.cu -- optional locality reorder of a loaded graph (QM_REORDER).
//
// Scoring gathers the label of every arc's far end.  With node ids in random
// order (as in the LFR benchmark graphs of Sec. IV-C, and in many real edge
// lists) those gathers land anywhere in the label array, which at 10^8 nodes
// is three times the L2 cache.  A partition worth scoring follows the graph's
// community structure, so renumbering the nodes cluster by cluster makes most
// of the gathered labels neighbours in memory.  The clusters come from the
// graph alone (a few synchronous label-propagation rounds, never from a
// partition being scored), the renumbering is done once when the graph is
// loaded, and each scoring call brings its labels into the stored order (a
// gather through the permutation, or on large graphs the two passes through
// shared memory at the end of this file).
// Every metric is invariant under renumbering and summed exactly, so the
// results are bit-identical with and without the reorder.
#include <algorithm>
#include <climits>
#include <cstdint>
#include <cstdio>

#include "qm_internal.h"
#include "qm_device.cuh"

namespace qm {

using namespace qmk;

// Labels start as the node ids.
__global__ void k_lpa_init(int *lab, long long n)
{
    for (long long u = (long long)blockIdx.x * blockDim.x + threadIdx.x; u < n; u += (long long)gridDim.x * blockDim.x)
        lab[u] = (int)u;
}

// One synchronous label-propagation round: a node takes the label found most
// often among (an evenly spaced sample of up to 32 of) its neighbours, keeps
// its own label when that is among the most frequent, and otherwise takes the
// smallest of the tied labels.
//
// A warp takes 32 consecutive nodes (fewer where those would not occupy the GPU,
// see lpa_shape).  First their samples one after another in
// slots, 32 slots a step whatever the degrees are (a bit per node's first slot
// and a popcount give a lane the node of its slot): a vote a step tells which
// labels equal the own one, and each node's lane then counts its bits.  A node
// with its own label in at least half of the sample keeps it (nothing can be more
// frequent).  The others are gathered LPA_NODES at a time, a lane per neighbour: the
// lanes match their labels and reduce (redux) the largest count, the own label
// counting half more, then the smallest label of that count.  In the first rounds
// hardly a node keeps its label, so those (`all`) skip the first part.
// Bound in the first rounds by the pipe of votes, matches and redux (80 % busy;
// DRAM 7 %), later by the gathers' latency.  Measured at 10^7 nodes (renumbered,
// mean degree 19, ten rounds), ms a call: a warp per node and a 64-bit shuffle
// reduction 14.2; a vote or two per node 8.62; so 7.79.  Steps in flight 2, 4, 8:
// 8.08, 7.87, 8.15; blocks per SM 5, 6, 7: 7.87, 7.87, 8.12; rounds with `all` 2
// and 3: 7.87, 7.79.
constexpr int LPA_NODES = 4;
constexpr int LPA_STEPS = 4;   // steps of 32 slots whose gathers are in flight together
constexpr int LPA_ALL_ROUNDS = 3;
constexpr int LPA_BLOCKS = 6;  // resident blocks per SM (40 registers), and those launched

struct LpaNode {
    long long at;   // first arc less the first slot; or (sampled) -1 - the first arc
    unsigned d, off;
};

template <int NODES>
__global__ void __launch_bounds__(256, LPA_BLOCKS) k_lpa_round(const long long *__restrict__ row_ptr, const int *__restrict__ col,
                                                   long long n, const int *__restrict__ cur, int *__restrict__ nxt,
                                                   int all)
{
    __shared__ LpaNode s_node[8][32];
    __shared__ int s_own[8][32];
    __shared__ unsigned s_first[8][32 + LPA_STEPS], s_eq[8][32 + LPA_STEPS + 1];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    LpaNode *const node = s_node[wid];
    int *const nown = s_own[wid];
    unsigned *const first_bits = s_first[wid], *const eq_bits = s_eq[wid];
    const long long nw = (long long)gridDim.x * (blockDim.x >> 5);
    for (long long u0 = (((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * NODES; u0 < n; u0 += nw * NODES) {
        const long long u = NODES == 32 || lane < NODES ? u0 + lane : n;
        const long long rs = __ldg(&row_ptr[min(u, n)]);
        const unsigned deg = (unsigned)(__ldg(&row_ptr[min(u + 1, n)]) - rs);  // 0 past the last node
        const int own = u < n ? __ldg(&cur[u]) : -1;
        const unsigned ds = min(deg, 32u);
        int res = own;
        unsigned wait;  // nodes not decided yet
        if (all) {
            wait = __ballot_sync(0xffffffffu, deg != 0u);
        } else {
            unsigned off = ds;
#pragma unroll
            for (int k = 1; k < 32; k <<= 1) {
                const unsigned t = __shfl_up_sync(0xffffffffu, off, k);
                if (lane >= k) off += t;
            }
            const unsigned total = __shfl_sync(0xffffffffu, off, 31);  // at most 1024
            off -= ds;
            const unsigned some = __ballot_sync(0xffffffffu, deg != 0u);
            first_bits[lane] = 0u;
            if (lane < LPA_STEPS) first_bits[32 + lane] = 0u;
            __syncwarp();
            if (deg) {
                const int k = __popc(some & ((1u << lane) - 1u));
                node[k] = deg <= 32u ? LpaNode{rs - (long long)off, 0u, 0u} : LpaNode{-1 - rs, deg, off};
                nown[k] = own;
                atomicOr(&first_bits[off >> 5], 1u << (off & 31u));
            }
            __syncwarp();
            int before = -1;  // nodes that began before this step, less one
            for (unsigned t0 = 0; t0 < total; t0 += 32u * LPA_STEPS) {
                int lab[LPA_STEPS], k[LPA_STEPS];
#pragma unroll
                for (int q = 0; q < LPA_STEPS; ++q) {
                    const unsigned m = first_bits[t0 / 32u + q], t = t0 + 32u * q + lane;
                    k[q] = max(before + __popc(m & (0xFFFFFFFFu >> (31 - lane))), 0);
                    before += __popc(m);
                    const LpaNode x = node[k[q]];
                    const long long a =
                        x.at >= 0 ? x.at + t : -1 - x.at + (long long)((unsigned long long)(t - x.off) * x.d / 32u);
                    lab[q] = t < total ? __ldg(&col[a]) : -1;
                }
#pragma unroll
                for (int q = 0; q < LPA_STEPS; ++q)
                    if (lab[q] >= 0) lab[q] = __ldg(&cur[lab[q]]);
#pragma unroll
                for (int q = 0; q < LPA_STEPS; ++q) {
                    const unsigned eq = __ballot_sync(0xffffffffu, lab[q] == nown[k[q]]);
                    if (lane == 0) eq_bits[t0 / 32u + q] = eq;
                }
            }
            __syncwarp();
            unsigned no = 0;
            if (ds) {
                const unsigned w = off >> 5;
                const unsigned b = __funnelshift_r(eq_bits[w], eq_bits[w + 1], off & 31u);
                no = __popc(b & (0xFFFFFFFFu >> (32u - ds)));
            }
            wait = __ballot_sync(0xffffffffu, 2u * no < ds);
            __syncwarp();
        }
        while (wait) {
            int lab[LPA_NODES], id[LPA_NODES];
#pragma unroll
            for (int q = 0; q < LPA_NODES; ++q) {
                id[q] = wait ? __ffs(wait) - 1 : -1;
                wait &= wait - 1u;
                const long long r = __shfl_sync(0xffffffffu, rs, id[q] & 31);
                const unsigned d = __shfl_sync(0xffffffffu, deg, id[q] & 31);
                const unsigned j = d <= 32u ? (unsigned)lane : (unsigned)((unsigned long long)lane * d / 32u);
                lab[q] = id[q] >= 0 && (unsigned)lane < d ? __ldcs(&col[r + j]) : -1;
            }
#pragma unroll
            for (int q = 0; q < LPA_NODES; ++q)
                if (lab[q] >= 0) lab[q] = __ldg(&cur[lab[q]]);
#pragma unroll
            for (int q = 0; q < LPA_NODES; ++q) {
                if (id[q] < 0) break;
                const int mine = __shfl_sync(0xffffffffu, own, id[q]);
                const unsigned peers = __match_any_sync(0xffffffffu, lab[q]);
                const unsigned c = lab[q] >= 0 ? 2u * (unsigned)__popc(peers) + (lab[q] == mine ? 1u : 0u) : 0u;
                const unsigned most = __reduce_max_sync(0xffffffffu, c);  // odd: the own label is among them
                int win = mine;
                if (!(most & 1u)) win = (int)__reduce_min_sync(0xffffffffu, c == most ? (unsigned)lab[q] : 0xFFFFFFFFu);
                if (lane == id[q]) res = win;
            }
        }
        if (u < n) nxt[u] = res;
    }
}

// Nodes per label.  Neighbours in the stored order mostly share theirs, so the
// first of each stretch of one label in a warp adds the stretch.
__global__ void k_count_ids(const int *__restrict__ lab, long long n, int *hist)
{
    const int lane = threadIdx.x & 31;
    const long long step = (long long)gridDim.x * blockDim.x;
    for (long long u0 = (long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31u); u0 < n; u0 += step) {
        const long long u = u0 + lane;
        const int x = u < n ? __ldg(&lab[u]) : -1;
        const int prev = __shfl_up_sync(0xffffffffu, x, 1);
        const unsigned heads = __ballot_sync(0xffffffffu, lane == 0 || x != prev);
        if (x >= 0 && ((heads >> lane) & 1u)) {
            const unsigned after = heads & (0xFFFFFFFEu << lane);
            atomicAdd(&hist[x], (after ? __ffs(after) - 1 : 32) - lane);
        }
    }
}

// New position of every node: its cluster's offset plus a slot taken in the
// cluster (the order inside a cluster is whatever the atomics give).
__global__ void k_place(const int *__restrict__ lab, long long n, int *cursor, int *inv, int *perm)
{
    for (long long u = (long long)blockIdx.x * blockDim.x + threadIdx.x; u < n;
         u += (long long)gridDim.x * blockDim.x) {
        const int pos = atomicAdd(&cursor[lab[u]], 1);
        inv[pos] = (int)u;
        perm[u] = pos;
    }
}

__global__ void k_new_degrees(const long long *__restrict__ row_ptr, const int *__restrict__ inv, long long n,
                              int *deg)
{
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (long long)gridDim.x * blockDim.x) {
        const int u = inv[j];
        deg[j] = (int)(row_ptr[u + 1] - row_ptr[u]);
    }
}

// 32-bit offsets (sum below 2^32) to the 64-bit row_ptr.
__global__ void k_widen(const unsigned *__restrict__ off, long long n, long long *row_ptr)
{
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j <= n; j += (long long)gridDim.x * blockDim.x)
        row_ptr[j] = (long long)off[j];
}

// Row j of the new CSR is row inv[j] of the old one with every neighbour
// renamed (and its weights, on a weighted graph); one warp per row.
__global__ void k_fill_rows(const long long *__restrict__ row_ptr, const int *__restrict__ col,
                            const int *__restrict__ inv, const int *__restrict__ perm, long long n,
                            const long long *__restrict__ row_ptr2, int *__restrict__ col2,
                            const float *__restrict__ wt, float *__restrict__ wt2)
{
    const int lane = threadIdx.x & 31;
    const long long nw = (long long)gridDim.x * (blockDim.x >> 5);
    for (long long j = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; j < n; j += nw) {
        const int u = __ldg(&inv[j]);
        const long long rs = __ldg(&row_ptr[u]), deg = __ldg(&row_ptr[u + 1]) - rs;
        const long long ws = __ldg(&row_ptr2[j]);
        for (long long e = lane; e < deg; e += 32) {
            col2[ws + e] = __ldg(&perm[__ldg(&col[rs + e])]);
            if (wt) wt2[ws + e] = __ldg(&wt[rs + e]);
        }
    }
}

// out[p][j] = labels[p][inv[j]] for P rows of n labels.
__global__ void k_permute_labels(const int *__restrict__ labels, const int *__restrict__ inv, long long n, int P,
                                 int *__restrict__ out)
{
    const long long total = n * (long long)P;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const long long p = i / n, j = i - p * n;
        out[i] = __ldg(&labels[p * n + __ldg(&inv[j])]);
    }
}

// Label propagation as a detector (qm_label_propagation): labels start as the
// caller's node ids, so a renumbered graph gives the same partition.
__global__ void k_lpa_init_ids(int *lab, const int *__restrict__ inv, long long n)
{
    for (long long u = (long long)blockIdx.x * blockDim.x + threadIdx.x; u < n; u += (long long)gridDim.x * blockDim.x)
        lab[u] = inv ? inv[u] : (int)u;
}

// flag[c] = 1 when some node carries label c (c in [0, n)).
__global__ void k_present(int *hist, long long n)
{
    for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x)
        hist[c] = hist[c] > 0 ? 1 : 0;
}

// out[caller id] = rank of the node's final label among the labels present.
__global__ void k_write_ranks(const int *__restrict__ lab, const int *__restrict__ rank, const int *__restrict__ inv,
                              long long n, int *__restrict__ out)
{
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (long long)gridDim.x * blockDim.x)
        out[inv ? inv[j] : j] = rank[lab[j]];
}

static int grid_of(long long work, int threads, int num_sms, int per_sm)
{
    long long g = (work + threads - 1) / threads;
    const long long cap = (long long)num_sms * per_sm;
    return (int)(g < 1 ? 1 : (g > cap ? cap : g));
}

// Nodes a warp of k_lpa_round takes, and its blocks.  Small graphs spread over the
// GPU: down to four nodes a warp where there are not four times as many
// warps as are resident.  Their labels are in L2 and the slots cost more than the
// matches they save, so all their rounds go without.  Ten rounds at 10^4, 10^5 and
// 6*10^5 nodes, mixing 0.5, us a call: a warp per node 126, 270, 1024; 32 nodes a
// warp with slots 211, 297, 997; so 127, 252, 870 (0.1: 129, 242, 899; 164, 210,
// 627; 126, 205, 627).  From 9*10^5 nodes on 32 (10^6 nodes, 0.1 and 0.5: a warp per
// node 1408 and 1619, 32 with slots 929 and 1538).
struct LpaShape {
    int nodes, grid;
    bool all(int round) const { return round < LPA_ALL_ROUNDS || nodes < 32; }
};

static LpaShape lpa_shape(long long n, int num_sms)
{
    LpaShape s{32, 0};
    while (s.nodes > 4 && n < 4LL * s.nodes * num_sms * LPA_BLOCKS * 8) s.nodes /= 2;
    s.grid = grid_of((n + s.nodes - 1) / s.nodes * 32, 256, num_sms, LPA_BLOCKS);
    return s;
}

static void launch_lpa_round(const GraphDev &g, const int *cur, int *nxt, int round, const LpaShape &s, cudaStream_t st)
{
    auto run = [&](auto kern) { kern<<<s.grid, 256, 0, st>>>(g.row_ptr, g.col, g.n, cur, nxt, s.all(round)); };
    if (s.nodes == 32) run(k_lpa_round<32>);
    else if (s.nodes == 16) run(k_lpa_round<16>);
    else if (s.nodes == 8) run(k_lpa_round<8>);
    else run(k_lpa_round<4>);
}

int launch_permute_labels(const int *labels, const int *inv, long long n, int P, int *out, int num_sms,
                          cudaStream_t s)
{
    k_permute_labels<<<grid_of(n * (long long)P, 512, num_sms, 8), 512, 0, s>>>(labels, inv, n, P, out);
    return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

int launch_label_propagation(const GraphDev &g, int rounds, int num_sms, cudaStream_t s, int *lab0, int *lab1,
                             int *hist, int *tmp, size_t tmp_elems, int *out)
{
    const long long n = g.n;
    const int g1 = grid_of(n, 512, num_sms, 8);
    const LpaShape ls = lpa_shape(n, num_sms);
    int L = 0;
    k_lpa_init_ids<<<g1, 512, 0, s>>>(lab0, g.inv, n);
    ++L;
    for (int r = 0; r < rounds; ++r) {
        launch_lpa_round(g, lab0, lab1, r, ls, s);
        std::swap(lab0, lab1);
        ++L;
    }
    if (cudaMemsetAsync(hist, 0, (size_t)(n + 1) * 4, s) != cudaSuccess) return -1;
    if (cudaMemsetAsync(tmp, 0, tmp_elems * 4, s) != cudaSuccess) return -1;
    k_count_ids<<<g1, 512, 0, s>>>(lab0, n, hist);
    k_present<<<g1, 512, 0, s>>>(hist, n);
    L += 2;
    int *status = tmp + tmp_elems - 32, *counters = tmp + tmp_elems - 16;
    const int l2 = scan_offsets(hist, (int)n, hist, tmp, counters, status, s);  // hist[n] = number of labels
    if (l2 < 0) return -1;
    L += l2;
    k_write_ranks<<<g1, 512, 0, s>>>(lab0, hist, g.inv, n, out);
    ++L;
    return cudaGetLastError() == cudaSuccess ? L : -1;
}

int reorder_graph(const GraphDev &g, int rounds, int num_sms, cudaStream_t s, long long **row_ptr_out, int **col_out,
                  int **inv_out, int *launches, float **wt_out)
{
    const long long n = g.n;
    int *lab0 = nullptr, *lab1 = nullptr, *hist = nullptr, *perm = nullptr, *inv = nullptr, *tmp = nullptr;
    long long *row2 = nullptr;
    int *col2 = nullptr;
    float *wt2 = nullptr;
    int L = 0;
    auto bad = [&](cudaError_t e) {
        cudaFree(lab0);
        cudaFree(lab1);
        cudaFree(hist);
        cudaFree(perm);
        cudaFree(inv);
        cudaFree(tmp);
        cudaFree(row2);
        cudaFree(col2);
        cudaFree(wt2);
        return e == cudaSuccess ? (int)cudaErrorUnknown : (int)e;
    };
    cudaError_t e = cudaSuccess;
    const size_t tmp_elems = scan_tmp_elems(n + 1) + 64;
    if ((e = cudaMalloc(&lab0, (size_t)n * 4)) != cudaSuccess) return -bad(e);
    if ((e = cudaMalloc(&lab1, (size_t)n * 4)) != cudaSuccess) return -bad(e);
    if ((e = cudaMalloc(&hist, (size_t)(n + 1) * 4)) != cudaSuccess) return -bad(e);
    if ((e = cudaMalloc(&perm, (size_t)n * 4)) != cudaSuccess) return -bad(e);
    if ((e = cudaMalloc(&inv, (size_t)n * 4)) != cudaSuccess) return -bad(e);
    if ((e = cudaMalloc(&tmp, tmp_elems * 4)) != cudaSuccess) return -bad(e);
    const int g1 = grid_of(n, 512, num_sms, 8), gw = grid_of(n * 32, 256, num_sms, 8);
    const LpaShape ls = lpa_shape(n, num_sms);
    k_lpa_init<<<g1, 512, 0, s>>>(lab0, n);
    ++L;
    for (int r = 0; r < rounds; ++r) {
        launch_lpa_round(g, lab0, lab1, r, ls, s);
        std::swap(lab0, lab1);
        ++L;
    }
    // cluster offsets: hist -> exclusive scan (in place, n + 1 entries) -> cursor
    if ((e = cudaMemsetAsync(hist, 0, (size_t)(n + 1) * 4, s)) != cudaSuccess) return -bad(e);
    if ((e = cudaMemsetAsync(tmp, 0, tmp_elems * 4, s)) != cudaSuccess) return -bad(e);
    k_count_ids<<<g1, 512, 0, s>>>(lab0, n, hist);
    ++L;
    int *status = tmp + tmp_elems - 32, *counters = tmp + tmp_elems - 16;
    int l2 = scan_offsets(hist, (int)n, hist, tmp, counters, status, s);
    if (l2 < 0) return -bad(cudaGetLastError());
    L += l2;
    k_place<<<g1, 512, 0, s>>>(lab0, n, hist, inv, perm);
    ++L;
    // new row offsets from the degrees in the new order (lab1 is free: reuse it)
    k_new_degrees<<<g1, 512, 0, s>>>(g.row_ptr, inv, n, lab1);
    ++L;
    l2 = scan_offsets(lab1, (int)n, hist, tmp, counters, status, s);
    if (l2 < 0) return -bad(cudaGetLastError());
    L += l2;
    if ((e = cudaMalloc(&row2, (size_t)(n + 1) * 8)) != cudaSuccess) return -bad(e);
    if ((e = cudaMalloc(&col2, (size_t)g.n_arcs * 4)) != cudaSuccess) return -bad(e);
    if (g.wt && (e = cudaMalloc(&wt2, (size_t)g.n_arcs * 4)) != cudaSuccess) return -bad(e);
    k_widen<<<g1, 512, 0, s>>>((const unsigned *)hist, n, row2);
    k_fill_rows<<<gw, 256, 0, s>>>(g.row_ptr, g.col, inv, perm, n, row2, col2, g.wt, wt2);
    L += 2;
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return -bad(e);
    if ((e = cudaGetLastError()) != cudaSuccess) return -bad(e);
    cudaFree(lab0);
    cudaFree(lab1);
    cudaFree(hist);
    cudaFree(perm);
    cudaFree(tmp);
    *row_ptr_out = row2;
    *col_out = col2;
    *inv_out = inv;
    if (wt_out) *wt_out = wt2;
    if (launches) *launches = L;
    return 0;
}

// ------------------------------------------------------------------ upper rows

// Arcs of node u to itself or to higher ids, one warp per row.
__global__ void k_up_degrees(const long long *__restrict__ row_ptr, const int *__restrict__ col, long long n,
                             int *deg)
{
    const int lane = threadIdx.x & 31;
    const long long nw = (long long)gridDim.x * (blockDim.x >> 5);
    for (long long u = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; u < n; u += nw) {
        const long long rs = __ldg(&row_ptr[u]), re = __ldg(&row_ptr[u + 1]);
        int cnt = 0;
        for (long long e = rs + lane; e < re; e += 32) cnt += __ldg(&col[e]) >= u ? 1 : 0;
        cnt = __reduce_add_sync(0xffffffffu, cnt);
        if (lane == 0) deg[u] = cnt;
    }
}

// Copies those arcs in row order, a self-loop as ~u; one warp per row.
__global__ void k_up_fill(const long long *__restrict__ row_ptr, const int *__restrict__ col, long long n,
                          const long long *__restrict__ up_ptr, int *__restrict__ up_col)
{
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const long long nw = (long long)gridDim.x * (blockDim.x >> 5);
    for (long long u = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; u < n; u += nw) {
        const long long rs = __ldg(&row_ptr[u]), re = __ldg(&row_ptr[u + 1]);
        long long at = __ldg(&up_ptr[u]);
        for (long long e0 = rs; e0 < re; e0 += 32) {
            const long long e = e0 + lane;
            const int v = e < re ? __ldg(&col[e]) : -1;
            const bool keep = e < re && v >= u;
            const unsigned m = __ballot_sync(0xffffffffu, keep);
            if (keep) up_col[at + __popc(m & lt)] = v == u ? ~v : v;
            at += __popc(m);
        }
    }
}

int build_upper_rows(const GraphDev &g, int num_sms, cudaStream_t s, long long **up_ptr_out, int **up_col_out,
                     long long *up_arcs, int *launches)
{
    const long long n = g.n;
    int *deg = nullptr, *tmp = nullptr;
    long long *up_ptr = nullptr;
    int *up_col = nullptr;
    unsigned *total_h = nullptr;
    auto bad = [&](cudaError_t e) {
        cudaFree(deg);
        cudaFree(tmp);
        cudaFree(up_ptr);
        cudaFree(up_col);
        cudaFreeHost(total_h);
        return e == cudaSuccess ? (int)cudaErrorUnknown : (int)e;
    };
    if (g.n_arcs >= (1LL << 32)) return -bad(cudaErrorInvalidValue);
    cudaError_t e = cudaSuccess;
    int L = 0;
    const size_t tmp_elems = scan_tmp_elems(n + 1) + 64;
    if ((e = cudaMalloc(&deg, (size_t)(n + 1) * 4)) != cudaSuccess) return -bad(e);
    if ((e = cudaMalloc(&tmp, tmp_elems * 4)) != cudaSuccess) return -bad(e);
    if ((e = cudaMalloc(&up_ptr, (size_t)(n + 1) * 8)) != cudaSuccess) return -bad(e);
    if ((e = cudaMallocHost(&total_h, 16)) != cudaSuccess) return -bad(e);
    if ((e = cudaMemsetAsync(tmp, 0, tmp_elems * 4, s)) != cudaSuccess) return -bad(e);
    const int g1 = grid_of(n, 512, num_sms, 8), gw = grid_of(n * 32, 256, num_sms, 8);
    k_up_degrees<<<gw, 256, 0, s>>>(g.row_ptr, g.col, n, deg);
    ++L;
    int *status = tmp + tmp_elems - 32, *counters = tmp + tmp_elems - 16;
    const int l2 = scan_offsets(deg, (int)n, deg, tmp, counters, status, s);  // deg[n] = total
    if (l2 < 0) return -bad(cudaGetLastError());
    L += l2;
    k_widen<<<g1, 512, 0, s>>>((const unsigned *)deg, n, up_ptr);
    ++L;
    if ((e = cudaMemcpyAsync(total_h, deg + n, 4, cudaMemcpyDeviceToHost, s)) != cudaSuccess) return -bad(e);
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return -bad(e);
    const long long total = (long long)total_h[0];
    if ((e = cudaMalloc(&up_col, (size_t)std::max(total, 1LL) * 4)) != cudaSuccess) return -bad(e);
    k_up_fill<<<gw, 256, 0, s>>>(g.row_ptr, g.col, n, up_ptr, up_col);
    ++L;
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return -bad(e);
    if ((e = cudaGetLastError()) != cudaSuccess) return -bad(e);
    cudaFree(deg);
    cudaFree(tmp);
    cudaFreeHost(total_h);
    *up_ptr_out = up_ptr;
    *up_col_out = up_col;
    if (up_arcs) *up_arcs = total;
    if (launches) *launches = L;
    return 0;
}

// ------------------------------------------------------------------ bucketed label permutation

// A scoring call on a renumbered graph first brings the caller's labels into
// the stored order, out[j] = labels[inv[j]].  As one gather that is a random
// 4-byte read per node from an array larger than L2, and each costs DRAM far
// more than 4 bytes.  The buckets built here do it in two passes whose global
// reads and writes are all sequential, the random part in shared memory:
//   pass 1  per tile of 2^tile_bits caller ids: the tile's labels are placed
//           in shared memory grouped by the window of 2^window_bits new ids
//           they are bound for, then each window's group is written to that
//           window's stretch of a scratch array (slots);
//   pass 2  per window: its slots are placed in shared memory at their new
//           ids, and the window is written out in order, the community sizes
//           counted on the way (labels of one cluster are adjacent then).
// Inside a (tile, window) group the order is whatever the build's atomics
// gave; both passes follow the same order, so the result does not depend on it.

constexpr int PB_BUILD_THREADS = 512;
constexpr int PB_THREADS = 1024;

__global__ void k_pb_invert(const int *__restrict__ inv, long long n, int *__restrict__ perm)
{
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (long long)gridDim.x * blockDim.x)
        perm[inv[j]] = (int)j;
}

// cnt[w * ntiles + t]: ids of tile t whose new id lies in window w.
__global__ void k_pb_count(const int *__restrict__ perm, long long n, int tb, int wb, int nw, int ntiles, int *cnt)
{
    extern __shared__ int c[];  // [nw]
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        for (int i = threadIdx.x; i < nw; i += blockDim.x) c[i] = 0;
        __syncthreads();
        const long long u0 = (long long)t << tb, u1 = min(n, u0 + (1LL << tb));
        for (long long u = u0 + threadIdx.x; u < u1; u += blockDim.x) atomicAdd(&c[perm[u] >> wb], 1);
        __syncthreads();
        for (int i = threadIdx.x; i < nw; i += blockDim.x) cnt[(long long)i * ntiles + t] = c[i];
        __syncthreads();
    }
}

// From the window-major exclusive prefix `off` (off[nw * ntiles] = n): per
// tile, toff[t][w] = first slot of group (t, w) and tlb[t][w] = its first
// position in the tile's grouped order (tlb[t][nw] = the tile's length).
__global__ void k_pb_tables(const int *__restrict__ off, int nw, int ntiles, int *toff, int *tlb)
{
    __shared__ int wsum[PB_BUILD_THREADS / 32];
    const int T = blockDim.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int per = (nw + T - 1) / T, w0 = min(nw, tid * per), w1 = min(nw, w0 + per);
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        int sum = 0;
        for (int w = w0; w < w1; ++w) {
            const long long i = (long long)w * ntiles + t;
            toff[(long long)t * nw + w] = off[i];
            sum += off[i + 1] - off[i];
        }
        int x = sum;  // inclusive scan over the block, chunk by chunk
        for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, d);
            if (lane >= d) x += y;
        }
        if (lane == 31) wsum[wid] = x;
        __syncthreads();
        if (wid == 0) {
            int v = lane < T / 32 ? wsum[lane] : 0;
            for (int d = 1; d < 32; d <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, v, d);
                if (lane >= d) v += y;
            }
            if (lane < T / 32) wsum[lane] = v;
        }
        __syncthreads();
        int run = x - sum + (wid > 0 ? wsum[wid - 1] : 0);
        for (int w = w0; w < w1; ++w) {
            const long long i = (long long)w * ntiles + t;
            tlb[(long long)t * (nw + 1) + w] = run;
            run += off[i + 1] - off[i];
        }
        if (tid == T - 1) tlb[(long long)t * (nw + 1) + nw] = wsum[T / 32 - 1];
        __syncthreads();
    }
}

// Each caller id's position in its tile's grouped order (lpos) and each
// slot's new id inside its window (dloc); ranks inside a group by atomics.
__global__ void k_pb_place(const int *__restrict__ perm, long long n, int tb, int wb, int nw, int ntiles,
                           const int *__restrict__ toff, const int *__restrict__ tlb, unsigned short *lpos,
                           unsigned short *dloc)
{
    extern __shared__ int cur[];  // [nw]
    const int mask = (1 << wb) - 1;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        for (int i = threadIdx.x; i < nw; i += blockDim.x) cur[i] = 0;
        __syncthreads();
        const long long u0 = (long long)t << tb, u1 = min(n, u0 + (1LL << tb));
        for (long long u = u0 + threadIdx.x; u < u1; u += blockDim.x) {
            const int j = perm[u], w = j >> wb;
            const int r = atomicAdd(&cur[w], 1);
            lpos[u] = (unsigned short)(tlb[(long long)t * (nw + 1) + w] + r);
            dloc[toff[(long long)t * nw + w] + r] = (unsigned short)(j & mask);
        }
        __syncthreads();
    }
}

// Shared memory of the passes with B bytes a label (3 while the labels are
// below 2^24, else 4).
static size_t pb_pass1_smem(int tb, int nw, int B) { return (size_t)B * ((size_t)1 << tb) + (2 * (size_t)nw + 1) * 4; }
static size_t pb_pass2_smem(int wb, int B) { return (size_t)B * ((size_t)1 << wb); }

// Whether the two passes fit with 3-byte labels: shared memory, 16-bit local
// positions, and tables of at most 2^30 entries.
static bool pb_fits(long long n, int wb, int tb, size_t smem_max, int *nw_out, int *ntiles_out)
{
    if (wb < 1 || wb > PB_MAX_BITS || tb < 1 || tb > PB_MAX_BITS) return false;
    const long long nw = (n + (1LL << wb) - 1) >> wb, ntiles = (n + (1LL << tb) - 1) >> tb;
    if (nw > PB_MAX_WINDOWS || nw * ntiles >= (1LL << 30)) return false;
    if (pb_pass1_smem(tb, (int)nw, 3) > smem_max || pb_pass2_smem(wb, 3) > smem_max) return false;
    *nw_out = (int)nw;
    *ntiles_out = (int)ntiles;
    return true;
}

template <int B, bool V4>
__global__ void k_pb_tile(const int *__restrict__ labels, const unsigned short *__restrict__ lpos,
                          const int *__restrict__ toff, const int *__restrict__ tlb, long long n, int tb, int nw,
                          int ntiles, int K, int *__restrict__ tmp, int *status);
template <int B, bool V4, bool SHARED>
__global__ void k_pb_window(const int *__restrict__ tmp, const unsigned short *__restrict__ dloc, long long n, int wb,
                            int nw, int *__restrict__ out, int *size, int K, const long long *__restrict__ row_ptr,
                            unsigned long long *cv, int counts_at);

template <int B, bool V4>
static cudaError_t pb_set_smem_v(size_t smem_max)
{
    cudaError_t e =
        cudaFuncSetAttribute(k_pb_tile<B, V4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_max);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_pb_window<B, V4, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_max);
    if (e == cudaSuccess && B == 3)  // (few ids are narrow)
        e = cudaFuncSetAttribute(k_pb_window<3, V4, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_max);
    return e;
}

template <int B>
static cudaError_t pb_set_smem(size_t smem_max)
{
    const cudaError_t e = pb_set_smem_v<B, false>(smem_max);
    return e == cudaSuccess ? pb_set_smem_v<B, true>(smem_max) : e;
}

int build_perm_buckets(const int *inv, long long n, int wb, int tb, int num_sms, cudaStream_t s, PermBuckets *out,
                       int *launches)
{
    int dev = 0, smem_optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return -(int)e;
    const size_t smem_max = (size_t)smem_optin;
    int nw = 0, ntiles = 0;
    if (!pb_fits(n, wb, tb, smem_max, &nw, &ntiles)) return 1;
    const long long ncnt = (long long)nw * ntiles;
    int *perm = nullptr, *cnt = nullptr, *tmp = nullptr, *toff = nullptr, *tlb = nullptr;
    unsigned short *lpos = nullptr, *dloc = nullptr;
    auto bad = [&](cudaError_t e) {
        cudaFree(perm);
        cudaFree(cnt);
        cudaFree(tmp);
        cudaFree(toff);
        cudaFree(tlb);
        cudaFree(lpos);
        cudaFree(dloc);
        return e == cudaSuccess ? (int)cudaErrorUnknown : (int)e;
    };
    const size_t tmp_elems = scan_tmp_elems(ncnt + 1) + 64;
    if ((e = cudaMalloc(&perm, (size_t)n * 4)) != cudaSuccess) return -bad(e);
    if ((e = cudaMalloc(&cnt, (size_t)(ncnt + 1) * 4)) != cudaSuccess) return -bad(e);
    if ((e = cudaMalloc(&tmp, tmp_elems * 4)) != cudaSuccess) return -bad(e);
    if ((e = cudaMalloc(&toff, (size_t)ncnt * 4)) != cudaSuccess) return -bad(e);
    if ((e = cudaMalloc(&tlb, (size_t)ntiles * (nw + 1) * 4)) != cudaSuccess) return -bad(e);
    if ((e = cudaMalloc(&lpos, (size_t)n * 2)) != cudaSuccess) return -bad(e);
    if ((e = cudaMalloc(&dloc, (size_t)n * 2)) != cudaSuccess) return -bad(e);
    if ((e = cudaMemsetAsync(tmp, 0, tmp_elems * 4, s)) != cudaSuccess) return -bad(e);
    if ((e = pb_set_smem<3>(smem_max)) != cudaSuccess || (e = pb_set_smem<4>(smem_max)) != cudaSuccess)
        return -bad(e);
    int L = 0;
    k_pb_invert<<<grid_of(n, 512, num_sms, 8), 512, 0, s>>>(inv, n, perm);
    const int gt = std::min(ntiles, num_sms * 4);
    k_pb_count<<<gt, PB_BUILD_THREADS, (size_t)nw * 4, s>>>(perm, n, tb, wb, nw, ntiles, cnt);
    L += 2;
    int *status = tmp + tmp_elems - 32, *counters = tmp + tmp_elems - 16;
    const int l2 = scan_offsets(cnt, (int)ncnt, cnt, tmp, counters, status, s);
    if (l2 < 0) return -bad(cudaGetLastError());
    L += l2;
    k_pb_tables<<<gt, PB_BUILD_THREADS, 0, s>>>(cnt, nw, ntiles, toff, tlb);
    k_pb_place<<<gt, PB_BUILD_THREADS, (size_t)nw * 4, s>>>(perm, n, tb, wb, nw, ntiles, toff, tlb, lpos, dloc);
    L += 2;
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return -bad(e);
    if ((e = cudaGetLastError()) != cudaSuccess) return -bad(e);
    cudaFree(perm);
    cudaFree(cnt);
    cudaFree(tmp);
    out->lpos = lpos;
    out->dloc = dloc;
    out->toff = toff;
    out->tlb = tlb;
    out->wb = wb;
    out->tb = tb;
    out->nw = nw;
    out->ntiles = ntiles;
    out->smem_max = smem_max;
    out->bytes = (size_t)n * 4 + (size_t)ncnt * 4 + (size_t)ntiles * (nw + 1) * 4;
    if (launches) *launches = L;
    return 0;
}

void free_perm_buckets(PermBuckets *pb)
{
    cudaFree(pb->lpos);
    cudaFree(pb->dloc);
    cudaFree(pb->toff);
    cudaFree(pb->tlb);
    *pb = PermBuckets{};
}

constexpr int PB_UNROLL = 4;

// A label in shared memory at position p, B bytes wide (little-endian; with
// B = 3 the labels are known to lie in [0, 2^24)).
template <int B>
__device__ __forceinline__ void pb_put(unsigned char *m, int p, int v)
{
    if (B == 4) {
        ((int *)m)[p] = v;
    } else {
        unsigned char *q = m + 3 * p;
        q[0] = (unsigned char)v;
        q[1] = (unsigned char)(v >> 8);
        q[2] = (unsigned char)(v >> 16);
    }
}

template <int B>
__device__ __forceinline__ int pb_get(const unsigned char *m, int p)
{
    if (B == 4) return ((const int *)m)[p];
    const unsigned char *q = m + 3 * p;
    return (int)q[0] | ((int)q[1] << 8) | ((int)q[2] << 16);
}

// Values v[0 .. len) into shared memory at positions pos[0 .. len), each
// checked against [0, K) (bad).  With V4, v and pos are 16- and 8-byte
// aligned and move four at a time, two groups in flight per thread.
template <int B, bool V4>
__device__ __forceinline__ void pb_stage(const int *__restrict__ v, const unsigned short *__restrict__ pos, int len,
                                         unsigned char *m, int K, bool &bad)
{
    const int T = blockDim.x, tid = threadIdx.x;
    int i = 0;
    if (V4) {
        const int ng = len >> 2;
        for (int g0 = 0; g0 < ng; g0 += 2 * T) {
            int4 x[2];
            ushort4 p[2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int g = g0 + q * T + tid;
                if (g < ng) {
                    x[q] = __ldcs((const int4 *)v + g);
                    p[q] = __ldcs((const ushort4 *)pos + g);
                }
            }
#pragma unroll
            for (int q = 0; q < 2; ++q)
                if (g0 + q * T + tid < ng) {
                    if ((unsigned)x[q].x >= (unsigned)K || (unsigned)x[q].y >= (unsigned)K ||
                        (unsigned)x[q].z >= (unsigned)K || (unsigned)x[q].w >= (unsigned)K)
                        bad = true;
                    pb_put<B>(m, p[q].x, x[q].x);
                    pb_put<B>(m, p[q].y, x[q].y);
                    pb_put<B>(m, p[q].z, x[q].z);
                    pb_put<B>(m, p[q].w, x[q].w);
                }
        }
        i = ng << 2;
    }
    for (int i0 = i; i0 < len; i0 += T * PB_UNROLL) {
        int x[PB_UNROLL], p[PB_UNROLL];
#pragma unroll
        for (int q = 0; q < PB_UNROLL; ++q) {
            const int k = i0 + q * T + tid;
            p[q] = k < len ? (int)__ldcs(&pos[k]) : -1;
            x[q] = k < len ? __ldcs(&v[k]) : 0;
        }
#pragma unroll
        for (int q = 0; q < PB_UNROLL; ++q)
            if (p[q] >= 0) {
                if ((unsigned)x[q] >= (unsigned)K) bad = true;
                pb_put<B>(m, p[q], x[q]);
            }
    }
}

// Pass 1, one tile per block step: labels into shared memory at their grouped
// positions (checked against [0, K): bit 0 of *status), then every (tile,
// window) group to its slots, a warp per group.
template <int B, bool V4>
__global__ void __launch_bounds__(PB_THREADS, 2) k_pb_tile(const int *__restrict__ labels,
                                                        const unsigned short *__restrict__ lpos,
                                                        const int *__restrict__ toff, const int *__restrict__ tlb,
                                                        long long n, int tb, int nw, int ntiles, int K,
                                                        int *__restrict__ tmp, int *status)
{
    extern __shared__ __align__(16) unsigned char smb[];
    int *lb = (int *)smb, *of = lb + nw + 1;
    unsigned char *sv = (unsigned char *)(of + nw);
    const int T = blockDim.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, W = T >> 5;
    bool bad = false;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const long long u0 = (long long)t << tb;
        const int len = (int)min(n - u0, 1LL << tb);
        for (int w = tid; w <= nw; w += T) lb[w] = tlb[(long long)t * (nw + 1) + w];
        for (int w = tid; w < nw; w += T) of[w] = toff[(long long)t * nw + w];
        pb_stage<B, V4>(labels + u0, lpos + u0, len, sv, K, bad);
        __syncthreads();
        for (int w = wid; w < nw; w += W) {
            const int b = lb[w], e = lb[w + 1], o = of[w];
            for (int k = b + lane; k < e; k += 32) tmp[o + (k - b)] = pb_get<B>(sv, k);
        }
        __syncthreads();
    }
    if (bad) atomicOr(status, 1);
}

// Pass 2, one window per block step: slots into shared memory at their new
// ids, then the window out in order.  With `size`, the labels are counted as
// k_hist does, with `cv` as k_permute_vol does (in shared memory from byte
// counts_at on with SHARED; pass 1 has checked the labels).
template <int B, bool V4, bool SHARED>
__global__ void __launch_bounds__(PB_THREADS, 1) k_pb_window(const int *__restrict__ tmp,
                                                          const unsigned short *__restrict__ dloc, long long n,
                                                          int wb, int nw, int *__restrict__ out, int *size, int K,
                                                          const long long *__restrict__ row_ptr,
                                                          unsigned long long *cv, int counts_at)
{
    extern __shared__ __align__(16) unsigned char smb[];
    const int T = blockDim.x, tid = threadIdx.x;
    unsigned *const shv = (unsigned *)(smb + counts_at);
    if (SHARED) vol_smem_zero(shv, K);
    for (int w = blockIdx.x; w < nw; w += gridDim.x) {
        const long long base = (long long)w << wb;
        const int len = (int)min(n - base, 1LL << wb);
        bool unused = false;
        pb_stage<B, V4>(tmp + base, dloc + base, len, smb, INT_MAX, unused);
        __syncthreads();
        for (int i0 = tid; i0 - (tid & 31) < len; i0 += T * PB_UNROLL) {  // warp-uniform trip count
            int l[PB_UNROLL];
            unsigned d[PB_UNROLL];
#pragma unroll
            for (int q = 0; q < PB_UNROLL; ++q) {
                const int i = i0 + q * T;
                l[q] = i < len ? pb_get<B>(smb, i) : -1;
                d[q] = cv && i < len ? (unsigned)(__ldg(&row_ptr[base + i + 1]) - __ldg(&row_ptr[base + i])) : 0u;
                if (i < len) out[base + i] = l[q];
            }
#pragma unroll
            for (int q = 0; q < PB_UNROLL; ++q) {
                const bool ok = (unsigned)l[q] < (unsigned)K;
                if (SHARED) {
                    vol_smem_add_warp(shv, K, l[q], d[q], ok);
                } else if (cv) {
                    vol_add_warp(cv, l[q], d[q], ok);
                } else if (size) {
                    const unsigned act = __ballot_sync(0xffffffffu, ok);
                    if (ok) {
                        const unsigned peers = __match_any_sync(act, l[q]);
                        if ((threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&size[l[q]], __popc(peers));
                    }
                }
            }
        }
        __syncthreads();
    }
    if (SHARED) vol_smem_flush(shv, K, cv);
}

int launch_permute_buckets(const int *labels, const PermBuckets &pb, const long long *row_ptr, long long n, int *tmp,
                           int *out, int *size, unsigned long long *cv, int K, int *status, int num_sms, cudaStream_t s, void (*tr)(const char *, cudaStream_t))
{
    const bool narrow = K <= (1 << 24);
    const int B = narrow ? 3 : 4;
    const size_t p1 = pb_pass1_smem(pb.tb, pb.nw, B), p2 = pb_pass2_smem(pb.wb, B);
    if (p1 > pb.smem_max || p2 > pb.smem_max) return 0;  // 4-byte labels do not fit: gather them instead
    const size_t at = (p2 + 15) / 16 * 16;  // the counters behind the window
    const bool counts = cv && K <= VOL_SMEM_IDS && at + (size_t)K * 8 <= pb.smem_max;
    const size_t p2c = counts ? at + (size_t)K * 8 : p2;
    // resident blocks per SM: two of PB_THREADS at most, and what shared memory allows
    auto per_sm = [](size_t smem) { return (int)std::max<size_t>(1, std::min<size_t>(2, 233472 / (smem + 1024))); };
    const int g1 = std::min(pb.ntiles, num_sms * per_sm(p1)), g2 = std::min(pb.nw, num_sms * per_sm(p2c));
    // four at a time where every tile (window) start keeps the 16-byte alignment
    const bool v1 = pb.tb >= 2 && ((uintptr_t)labels & 15) == 0, v2 = pb.wb >= 2;
    auto pass1 = [&](auto kern) {
        kern<<<g1, PB_THREADS, p1, s>>>(labels, pb.lpos, pb.toff, pb.tlb, n, pb.tb, pb.nw, pb.ntiles, K, tmp, status);
    };
    auto pass2 = [&](auto kern) {
        kern<<<g2, PB_THREADS, p2c, s>>>(tmp, pb.dloc, n, pb.wb, pb.nw, out, size, K, row_ptr, cv, (int)at);
    };
    if (tr) tr("k_pb_tile", s);
    if (narrow)
        v1 ? pass1(k_pb_tile<3, true>) : pass1(k_pb_tile<3, false>);
    else
        v1 ? pass1(k_pb_tile<4, true>) : pass1(k_pb_tile<4, false>);
    if (tr) tr("k_pb_window", s);
    if (counts) v2 ? pass2(k_pb_window<3, true, true>) : pass2(k_pb_window<3, false, true>);
    else if (narrow) v2 ? pass2(k_pb_window<3, true, false>) : pass2(k_pb_window<3, false, false>);
    else v2 ? pass2(k_pb_window<4, true, false>) : pass2(k_pb_window<4, false, false>);
    return cudaGetLastError() == cudaSuccess ? 2 : -1;
}

}  // namespace qm
