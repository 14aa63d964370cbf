// Counts one run with one warp in a build with -DQM_BOUNDS_CHECK, one of whose
// labels is out of range: for tests/test_gpu_bounds_check.py.
#include "qm_count.cuh"

using namespace qmk;

template <int MODE>
__global__ void k_run(CountCtx x, RunHdr h)
{
    __shared__ __align__(16) unsigned slot[CT_WORDS];
    __shared__ unsigned late[CT_LATE];
    __shared__ unsigned long long red[8];
    for (int i = threadIdx.x; i < CT_WORDS; i += 32) slot[i] = 0u;
    __syncwarp();
    ct_count_run<MODE, false, 32>(x, h, x.nbr, slot, ct_count_bits(x.K), threadIdx.x, late, red);
}

// labels: m device ints; recip: K device reciprocals (2 words each); inter, rec:
// K zeroed ints and 8 K zeroed words; dbg: 8 host words.  Returns a CUDA error.
extern "C" int checked_run(int mode, const int *labels, int m, int K, const void *recip, int *inter,
                           unsigned long long *rec, unsigned long long *dbg)
{
    CountCtx x{};
    x.nbr = labels;
    x.inter = inter;
    x.recip = (const Rcp *)recip;
    x.rec = rec;
    x.K = K;
    const RunHdr h{0, 0u, (unsigned)m, (unsigned)m};
    const unsigned long long zero[8] = {};
    cudaMemcpyToSymbol(qm_dbg_rec, zero, sizeof zero);
    if (mode == CT_ABOVE) k_run<CT_ABOVE><<<1, 32>>>(x, h);
    else k_run<CT_FULL><<<1, 32>>>(x, h);
    const cudaError_t e = cudaDeviceSynchronize();
    cudaMemcpyFromSymbol(dbg, qm_dbg_rec, sizeof zero);
    return (int)e;
}
