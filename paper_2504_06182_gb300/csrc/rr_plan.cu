// rr_plan.cu -- kernels of the red-rec planner (arXiv 2504.06182, Alg. 1):
// each runs one stage of rr_plan.cuh over the instance array, blockIdx.y
// selecting the instance (blockIdx.x for the one-block-per-instance stages);
// `per` warps of a block on each instance where a warp takes an item.
#include "rr_plan.cuh"

namespace rrk {

__global__ void k_plan_setup(rr_instance *inst, JobWS *wsv, int count, int max_side, Arena A)
{
    s_plan_setup(hw_blk(), inst, wsv, count, max_side, A);
}

// Planning of one grid begins: its descriptor arrives as a kernel parameter
// (no copy before it) and the arena starts afresh.
__global__ void k_plan_begin(rr_instance h, rr_instance *I, JobWS *ws, int max_side, Arena A)
{
    if (threadIdx.x == 0) { *I = h; *A.top = 0; }
    __syncthreads();
    s_plan_setup(hw_blk(), I, ws, 1, max_side, A);
}

// Red-rec planning of one small grid by one block, block barriers instead of
// kernel boundaries (the single-grid kernel without bird and batching).
__global__ void __launch_bounds__(256) k_plan_block(rr_instance h, rr_instance *I, JobWS *ws, Arena A, int side)
{
    const int wid = threadIdx.x >> 5;
    const Blk B{0, 0, 1, wid, 8};
    if (threadIdx.x == 0) { *I = h; *A.top = 0; }
    __syncthreads();
    s_plan_setup(B, I, ws, 1, side, A);
    __syncthreads();
    s_transpose(B, I, ws, 1);
    __syncthreads();
    s_colstats(B, I, ws, 1, 0);
    __syncthreads();
    if (wid == 0) s_pair(B, I, ws, 1, 1);
    __syncthreads();
    s_emit_cols(B, I, ws, 1);
    s_emit_recv(B, I, ws, 1);
}

__global__ void k_transpose(rr_instance *inst, JobWS *wsv, int count, int per)
{
    s_transpose(hw_blk_shared(per), inst, wsv, count);
}

__global__ void k_colstats(rr_instance *inst, JobWS *wsv, int count, int strict, int per)
{
    s_colstats(hw_blk_shared(per), inst, wsv, count, strict);
}

// Lists an instance that has receiver units, once it is paired, for
// k_emit_recv. (It costs the pairing loop's code 1.5 %, so that calls over few
// grids, whose time that loop is, go without.)
__device__ __forceinline__ void list_lacking(const rr_instance *inst, JobWS *wsv, int q)
{
    if ((threadIdx.x & 31) == 0 && live(&inst[q]) && wsv[q].nrecv > 0)
        wsv[atomicAdd(&wsv[0].nlacking, 1)].lacking = q;
}

__global__ void k_pair(rr_instance *inst, JobWS *wsv, int count, int warm)
{
    s_pair(hw_blk(), inst, wsv, count, warm);
}

__global__ void k_pair_many(rr_instance *inst, JobWS *wsv, int count)
{
    s_pair(hw_blk(), inst, wsv, count, 0);
    list_lacking(inst, wsv, blockIdx.x);
}

__global__ void k_pair_sift(rr_instance *inst, JobWS *wsv, int count)
{
    s_pair_sift(hw_blk(), inst, wsv, count);
}

__global__ void k_pair_listed(rr_instance *inst, JobWS *wsv, int count)
{
    const int n = wsv[0].npending;
    Blk B = hw_blk();
    for (int i = blockIdx.x; i < n; i += gridDim.x) {
        B.x = wsv[i].pending;
        s_pair(B, inst, wsv, count, 0);
        list_lacking(inst, wsv, B.x);
        __syncwarp();
    }
}

__global__ void k_emit_cols(rr_instance *inst, JobWS *wsv, int count, int per)
{
    s_emit_cols(hw_blk_shared(per), inst, wsv, count);
}

// (more resident warps are worth more here than registers: 95 of them left
// room for 16 warps per SM)
// The launch's warps are shared out among the instances, in calls over many
// grids among those that have receiver units: how many these are, the host
// cannot know (1D chains have none, and eleven idle blocks for each took 10 of
// the 71 us of a call over 700 of them). The last to be paired come first: they
// have the most units (2 000 grids of sides 33 to 251: 315 us with four blocks
// each, 268 this way).
__global__ void __launch_bounds__(256, 5) k_emit_recv(rr_instance *inst, JobWS *wsv, int count, int listed)
{
    const int n = listed ? wsv[0].nlacking : count;
    if (n == 0) return;
    const int nw = (int)gridDim.x * 8 / n, g = (int)blockIdx.x * 8 + (int)(threadIdx.x >> 5), i = g / nw;
    if (i < n) s_emit_recv(Blk{0, listed ? wsv[n - 1 - i].lacking : i, 1, g % nw, nw}, inst, wsv, count);
}

int guard_cap_plan(long long cap)
{
    return cudaMemcpyToSymbol(g_guard_cap, &cap, sizeof(cap)) == cudaSuccess ? RR_OK : RR_ERR_CUDA;
}

} // namespace rrk
