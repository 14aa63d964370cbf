// qm_finalize.cuh -- from exact sums to the metric values (shared by the plain
// and the batched kernels so that both produce bit-identical results).
#pragma once

#include "qm_device.cuh"
#include "../../include/qm.h"

namespace qmk {

// Words of a partition's sums, written by lane 0 of a warp from the 32 lanes'
// accumulators: three 43-bit limbs per 128-bit sum, so that words of several
// warps and blocks add up as plain 64-bit integers.
__device__ __forceinline__ void score_words_warp(const ScoreAcc &acc, i128 qw, unsigned long long *w)
{
    const bool first = (threadIdx.x & 31u) == 0u;
    const i128 v[8] = {acc.qds_self, acc.qds_pair, acc.dens, acc.contr, acc.expn, acc.cond, (i128)acc.vol2, qw};
    const int at[8] = {GS_QDS_SELF, GS_QDS_PAIR, GS_DENS, GS_CONTR, GS_EXPN, GS_COND, GS_VOL2, GS_QW};
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const i128 t = warp_sum_i128_redux(v[k]);
        if (first) limbs_store(w + at[k], t);
    }
    const unsigned long long u[5] = {acc.ein, acc.eout, acc.nonempty, acc.slots, acc.cnt2};
    const int au[5] = {GS_EIN, GS_EOUT, GS_NONEMPTY, GS_SLOTS, GS_CNT2};
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const unsigned long long t = warp_sum_u64_redux(u[k]);
        if (first) w[au[k]] = t;
    }
}

__device__ __forceinline__ void compare_words_warp(const CompareAcc &acc, unsigned long long *w)
{
    const bool first = (threadIdx.x & 31u) == 0u;
    const i128 v[4] = {acc.vi, acc.hnum, acc.hden, acc.f};
    const int at[4] = {GC_VI, GC_HNUM, GC_HDEN, GC_F};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const i128 t = warp_sum_i128_redux(v[k]);
        if (first) limbs_store(w + at[k], t);
    }
    const unsigned long long u[7] = {acc.a11, acc.sa, acc.sb, acc.nvd, acc.cells, acc.ka, acc.kb};
    const int au[7] = {GC_A11, GC_SA, GC_SB, GC_NVD, GC_CELLS, GC_KA, GC_KB};
#pragma unroll
    for (int k = 0; k < 7; ++k) {
        const unsigned long long t = warp_sum_u64_redux(u[k]);
        if (first) w[au[k]] = t;
    }
}

// The same words from one thread's accumulators (weighted sums apart).
__device__ __forceinline__ void score_words(const ScoreAcc &a, unsigned long long *w)
{
    limbs_store(w + GS_QDS_SELF, a.qds_self);
    limbs_store(w + GS_QDS_PAIR, a.qds_pair);
    limbs_store(w + GS_DENS, a.dens);
    limbs_store(w + GS_CONTR, a.contr);
    limbs_store(w + GS_EXPN, a.expn);
    limbs_store(w + GS_COND, a.cond);
    limbs_store(w + GS_VOL2, (i128)a.vol2);
    w[GS_EIN] = a.ein;
    w[GS_EOUT] = a.eout;
    w[GS_NONEMPTY] = a.nonempty;
    w[GS_SLOTS] = a.slots;
    w[GS_CNT2] = a.cnt2;
}

__device__ __forceinline__ void compare_words(const CompareAcc &a, unsigned long long *w)
{
    limbs_store(w + GC_VI, a.vi);
    limbs_store(w + GC_HNUM, a.hnum);
    limbs_store(w + GC_HDEN, a.hden);
    limbs_store(w + GC_F, a.f);
    w[GC_A11] = a.a11;
    w[GC_SA] = a.sa;
    w[GC_SB] = a.sb;
    w[GC_NVD] = a.nvd;
    w[GC_CELLS] = a.cells;
    w[GC_KA] = a.ka;
    w[GC_KB] = a.kb;
}

__device__ __forceinline__ double i128_to_double(i128 v) { return fp_to_double(v, 0); }

// From exact sums to the metric values, by one warp with its 32 lanes: every
// value is one quotient, and lane k forms the k-th.  A chain of the eight
// divisions in one thread costs some 6 us, FP64 latency being what it is here.

// Eqs. (8), (9) and the Sec. II-B.3 means from the GS_* words g (readable by
// every lane).
//   Q = sum_c [E_in/|E| - (vol_c/(2|E|))^2] = (4|E| sum E_in - sum vol_c^2) / (4|E|^2),
// evaluated from exact integers with one rounding of numerator and denominator
// (weighted: the sum of the communities' terms).
__device__ __forceinline__ void quality_warp(const unsigned long long *g, long long n, long long E, bool weighted,
                                             qm_quality *out)
{
    const int lane = threadIdx.x & 31;
    const int at = lane == 0 ? GS_DENS : lane == 1 ? GS_CONTR : lane == 2 ? GS_EXPN : lane == 3 ? GS_COND
                   : lane == 4 ? GS_QDS_SELF : weighted ? GS_QW : GS_VOL2;
    i128 v = limbs_get(g + at);
    if (lane == 4) v -= limbs_get(g + GS_QDS_PAIR);
    if (lane == 5 && !weighted) v = (i128)4 * (i128)E * (i128)g[GS_EIN] - v;
    if (lane == 6) v = (i128)g[GS_EIN];
    if (lane == 7) v = (i128)g[GS_EOUT];
    const int scale = lane < 4 ? SC_MEAN : lane == 4 || (lane == 5 && weighted) ? SC_QDS : 0;
    const double d = lane == 4 || (lane == 5 && weighted) ? 1.0  // (a quotient by one is the value itself)
                     : lane == 5 ? i128_to_double((i128)4 * (i128)E * (i128)E)
                                 : (double)g[GS_NONEMPTY];
    const double r = __ddiv_rn(fp_to_double(v, scale), d);
    switch (lane) {
    case 0: out->mean_intra_density = r; break;
    case 1: out->mean_contraction = r; break;
    case 2: out->mean_expansion = r; break;
    case 3: out->mean_conductance = r; break;
    case 4: out->modularity_density = r; break;
    case 5: out->modularity = r; break;
    case 6: out->mean_intra_edges = r; break;
    case 7: out->mean_inter_edges = r; break;
    case 8:
        out->n_nodes = n;
        out->n_edges = E;
        out->n_communities_nonempty = (long long)g[GS_NONEMPTY];
        out->intra_edges_total = (long long)g[GS_EIN];
        out->cut_edges_total = (long long)(g[GS_EOUT] / 2);
        out->n_community_pairs = (long long)g[GS_SLOTS];  // each unordered pair counted once
        out->pair_count_sq_sum = (long long)g[GS_CNT2];
        break;
    default: break;
    }
}

// Eqs. (1)-(7) from the GC_* words g.  Pair counts of Sec. II-A.3 from the
// contingency table:
//   a11 = sum C(n_cc', 2), a11 + a10 = sum C(|c|, 2) = S_a, a11 + a01 = S_b,
//   A = C(N, 2).  RI, JI and ARI are ratios of exact integers; ARI is Eq. (6)
//   multiplied through by 2A: 2(A a11 - S_a S_b) / (A (S_a + S_b) - 2 S_a S_b).
__device__ __forceinline__ void compare_warp(const unsigned long long *g, long long N, qm_compare *out)
{
    const int lane = threadIdx.x & 31;
    const long long A = N * (N - 1) / 2;
    const long long a11 = (long long)g[GC_A11];
    const long long a10 = (long long)g[GC_SA] - a11;
    const long long a01 = (long long)g[GC_SB] - a11;
    const long long a00 = A - a11 - a10 - a01;
    const i128 sa = (i128)g[GC_SA], sb = (i128)g[GC_SB], a = (i128)A;
    const int at = lane == 0 ? GC_VI : lane == 1 ? GC_HNUM : GC_F;
    i128 v = limbs_get(g + at), w = (i128)N;
    int vs = lane == 0 ? SC_VI : lane == 1 ? SC_H : SC_F, ws = 0;
    bool one = false;  // 0 / 0: the value is 1
    if (lane == 1) {
        w = limbs_get(g + GC_HDEN);
        ws = SC_H;
        one = w == 0;
    } else if (lane == 3) {
        v = (i128)g[GC_NVD];
        vs = 0;
    } else if (lane == 4) {
        v = (i128)(a11 + a00);
        w = a;
        vs = 0;
    } else if (lane == 5) {
        v = 2 * (a * (i128)a11 - sa * sb);
        w = a * (sa + sb) - 2 * sa * sb;
        vs = 0;
        one = w == 0;
    } else if (lane == 6) {
        v = (i128)a11;
        w = (i128)(a11 + a10 + a01);
        vs = 0;
        one = w == 0;
    }
    double num = fp_to_double(v, vs), den = fp_to_double(w, ws);
    if (lane == 1) num = __dmul_rn(-2.0, num);
    if (lane == 3) den = __dmul_rn(2.0, den);
    const double r = one ? 1.0 : __ddiv_rn(num, den);
    switch (lane) {
    case 0: out->vi = -r; break;
    case 1: out->nmi = r; break;
    case 2: out->f_measure = r; break;
    case 3: out->nvd = __dsub_rn(1.0, r); break;
    case 4: out->ri = r; break;
    case 5: out->ari = r; break;
    case 6: out->ji = r; break;
    case 7:
        out->n_nodes = N;
        out->k_truth = (long long)g[GC_KA];
        out->k_found = (long long)g[GC_KB];
        out->n_cells = (long long)g[GC_CELLS];
        out->a11 = a11;
        out->a10 = a10;
        out->a01 = a01;
        out->a00 = a00;
        out->nvd_sum = (long long)g[GC_NVD];
        break;
    default: break;
    }
}

}  // namespace qmk
