// rr_batch.cu -- kernels of the batching routine (arXiv 2504.06182, Alg. 4
// with the local constraint set of Sec. IV): each runs one stage of
// rr_batch.cuh over the instance array.
#include "rr_batch.cuh"

namespace rrk {

// Batching of one move list begins: its descriptor arrives as a kernel
// parameter and the arena starts afresh.
__global__ void k_batch_begin(rr_instance h, rr_instance *I, Arena A)
{
    if (threadIdx.x == 0) { *I = h; *A.top = 0; }
}

__global__ void k_bsetup(rr_instance *inst, JobWS *wsv, int count, int max_side, Arena A, int lookback)
{
    s_bsetup(hw_blk(), inst, wsv, count, max_side, A, lookback);
}

__global__ void __launch_bounds__(LB_THREADS) k_pairoff_lookback(rr_instance *inst, JobWS *wsv, int count, Arena A)
{
    s_pairoff_lookback(hw_blk(), inst, wsv, count, A);
}

__global__ void k_gcount(rr_instance *inst, JobWS *wsv, int count)
{
    s_gcount(hw_blk(), inst, wsv, count);
}

__global__ void k_gscan(rr_instance *inst, JobWS *wsv, int count)
{
    s_gscan(hw_blk(), inst, wsv, count);
}

__global__ void k_gfill(rr_instance *inst, JobWS *wsv, int count)
{
    s_gfill(hw_blk(), inst, wsv, count);
}

__global__ void k_gsort(rr_instance *inst, JobWS *wsv, int count, int bufLen)
{
    s_gsort(hw_blk(), inst, wsv, count, bufLen);
}

__global__ void k_gsweep_h(rr_instance *inst, JobWS *wsv, int count, int lineCap)
{
    s_gsweep_h(hw_blk(), inst, wsv, count, lineCap);
}

__global__ void k_gsweep_v(rr_instance *inst, JobWS *wsv, int count, int lineCap)
{
    s_gsweep_v(hw_blk(), inst, wsv, count, lineCap);
}

__global__ void k_bsucc(rr_instance *inst, JobWS *wsv, int count)
{
    s_bsucc(hw_blk(), inst, wsv, count);
}

__global__ void k_bnum(rr_instance *inst, JobWS *wsv, int count)
{
    s_bnum(hw_blk(), inst, wsv, count);
}

__global__ void k_brec(rr_instance *inst, JobWS *wsv, int count)
{
    s_brec(hw_blk(), inst, wsv, count);
}

__global__ void k_order(const rr_instance *inst, int count, int *perm)
{
    s_order(hw_blk(), inst, count, perm);
}

__global__ void k_gather(const rr_instance *inst, const int *perm, rr_instance *pinst)
{
    s_gather(hw_blk(), inst, perm, pinst);
}

__global__ void k_scatter(rr_instance *inst, const int *perm, const rr_instance *pinst, int count)
{
    s_scatter(hw_blk(), inst, perm, pinst, count);
}

__global__ void k_classify(rr_instance *inst, int count, int nclass, int max_side, int *classCount,
                           int *classList)
{
    s_classify(hw_blk(), inst, count, nclass, max_side, classCount, classList);
}

// The simulation: one block per instance (of a size class's list, or of the
// whole call).
template <int MODE, bool WRITERS>
__device__ __forceinline__ void sim_of_block(rr_instance *inst, JobWS *wsv, int count, const int *classList,
                                             const int *classCount, int side, int counters)
{
    extern __shared__ int4 sim_smem[];
    int q = blockIdx.x;
    if (classList) {
        if (q >= *classCount) return;
        q = classList[q];
    }
    if (q >= count) return;
    sim_block<MODE, WRITERS>(&inst[q], wsv[q], (char *)sim_smem, side, counters);
}

// One warp, sides up to 256 and beyond; the same with writers. (A register
// too few costs more than a block too few per SM: with 96 instead of 128
// registers a 256 x 256 grid took 22 instead of 18 ms.)
#define SIM_KERNEL(name, mode, writers, threads, blocks)                                                      \
    __global__ void __launch_bounds__(threads, blocks) name(rr_instance *inst, JobWS *wsv, int count,         \
                                                            const int *classList, const int *classCount,      \
                                                            int side, int counters)                           \
    {                                                                                                         \
        sim_of_block<mode, writers>(inst, wsv, count, classList, classCount, side, counters);                 \
    }
SIM_KERNEL(k_sim, SIM_SMALL, false, 32, SIM_BLOCKS)
SIM_KERNEL(k_sim_big, SIM_BIG, false, 32, 12)
SIM_KERNEL(k_simw, SIM_SMALL, true, SIM_MAX_THREADS, 2)
SIM_KERNEL(k_simw_big, SIM_BIG, true, SIM_MAX_THREADS, 2)

// The simulations without writers that outgrew their tables.
__global__ void __launch_bounds__(32) k_sim_wide(rr_instance *inst, JobWS *wsv, int count, const int *classList,
                                                 const int *classCount, int side)
{
    extern __shared__ int4 wide_smem[];
    int q = blockIdx.x;
    if (classList) {
        if (q >= *classCount) return;
        q = classList[q];
    }
    if (q < count) s_wide(&inst[q], wsv[q], (char *)wide_smem, side);
}

// The batches of simulations that ran without writers.
__global__ void __launch_bounds__(256, 6) k_write(rr_instance *inst, JobWS *wsv, int count, const int *classList,
                                                  const int *classCount, int side)
{
    extern __shared__ int32_t write_smem[];
    int q = blockIdx.y;
    if (classList) {
        if (q >= *classCount) return;
        q = classList[q];
    }
    if (q >= count) return;
    s_write(hw_blk(), &inst[q], wsv[q], write_smem + sim_pow2(side) * (threadIdx.x >> 5));
}

int guard_cap_batch(long long cap)
{
    return cudaMemcpyToSymbol(g_guard_cap, &cap, sizeof(cap)) == cudaSuccess ? RR_OK : RR_ERR_CUDA;
}

} // namespace rrk
