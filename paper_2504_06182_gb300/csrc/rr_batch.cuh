// rr_batch.cuh -- stages of the batching routine (arXiv 2504.06182, Alg. 4 with the
// local constraint set of Sec. IV) on the GPU.
//
// Gamma (Sec. IV, "Input to the batching routine"): move b depends on every
// earlier move whose path shares a vertex with it. It is enough to keep, for
// every vertex, the immediately preceding path through it; a move is ready
// once all of those have finished. The kernels below build, per vertex, the
// list of paths through it in id order, and from it the de-duplicated
// successor lists and in-degrees.
//
// Alg. 4 itself runs as an event-driven simulation (below).
#pragma once
#include "rr_internal.cuh"

namespace rrk {

// Chunked block-wide exclusive scan of v[0..len) in place; returns the total.
// Every thread of the block must call it.
__device__ inline long long block_exclusive_scan(int32_t *v, int len, long long *s_tmp /* >= 33 */)
{
    const int T = blockDim.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int per = (len + T - 1) / T;
    const int lo = min(len, tid * per), hi = min(len, lo + per);
    long long sum = 0;
    for (int i = lo; i < hi; ++i) sum += v[i];
    long long incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        long long u = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += u;
    }
    if (lane == 31) s_tmp[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        long long w = lane < (T >> 5) ? s_tmp[lane] : 0;
        long long wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            long long u = __shfl_up_sync(FULL, wi, o);
            if (lane >= o) wi += u;
        }
        if (lane < (T >> 5)) s_tmp[lane] = wi - w;
        if (lane == 31) s_tmp[32] = wi;
    }
    __syncthreads();
    long long run = s_tmp[wid] + incl - sum;
    for (int i = lo; i < hi; ++i) { const long long x = v[i]; v[i] = (int32_t)run; run += x; }
    const long long total = s_tmp[32];
    __syncthreads();
    return total;
}

// ----------------------------------------------------------- set-up pass
// One block per instance: check the moves, count path vertices, allocate.
// An instance whose sizes the launch's shared memory does not cover (or that
// carries no list) ends here: with RR_BATCH_ONLY no planning kernel has looked
// at it, and every later stage indexes by its m, n and n_moves.
__device__ inline void s_bsetup(const Blk B, rr_instance *inst, JobWS *wsv, int count, int max_side, Arena A, int lookback)
{
    __shared__ long long s_tmp[34];
    __shared__ int s_bad;
    const int q = B.x;
    if (q >= count) return;
    rr_instance *I = &inst[q];
    if (!live(I)) return;
    JobWS &ws = wsv[q];
    const int m = I->m, n = I->n;
    const int64_t k = I->n_moves;
    if (m < 1 || n < 1 || m > max_side || n > max_side || k < 0 || k > 0x3fffffff || (k > 0 && !I->moves)) {
        __syncthreads();                    // (every thread has read the status)
        if (threadIdx.x == 0) I->status = RR_ERR_ARG;
        return;
    }
    if (lookback && k >= LB_MIN_MOVES) {
        // a large move list: checking the moves, counting their vertices and
        // the offsets are the work of the multi-block k_pairoff_lookback,
        // which also allocates the vertex-sized arrays once the total is
        // known; here only the move-sized arrays
        __shared__ int s_ok;
        if (threadIdx.x == 0) {
            bool ok = true;
            const unsigned long long cells = (unsigned long long)m * n;
            ws.P = -1;
            ws.pairOff = (int32_t *)arena_alloc(A, 4ull * (k + 1), &ok);
            ws.colOff = (int32_t *)arena_alloc(A, 4ull * (n + 1), &ok);
            ws.colCur = (int32_t *)arena_alloc(A, 4ull * (n + 1), &ok);
            ws.colList = (int32_t *)arena_alloc(A, 4ull * (k + 1), &ok);
            ws.rowOff = (int32_t *)arena_alloc(A, 4ull * (m + 1), &ok);
            ws.rowCur = (int32_t *)arena_alloc(A, 4ull * (m + 1), &ok);
            ws.rowList = (int32_t *)arena_alloc(A, 4ull * (k + 1), &ok);
            ws.firstH = (int32_t *)arena_alloc(A, 4ull * cells, &ok);
            ws.multiMove = (int2 *)arena_alloc(A, 8ull * (k + 1), &ok);
            ws.indeg = (int32_t *)arena_alloc(A, 4ull * (k + 1), &ok);
            ws.rec = (int4 *)arena_alloc(A, 32ull * (k + 1), &ok);
            ws.ready0 = (int32_t *)arena_alloc(A, 4ull * (k + 1) + 16, &ok);
            ws.state = (int2 *)arena_alloc(A, sim_wide_bytes(k), &ok);
            ws.multi = ws.colList;               // both lists are free again once they have been swept
            ws.multiNo = ws.rowList;
            ws.nmulti = 0;
            ws.nextAt = nullptr;
            ws.succ = nullptr;
            ws.lbStatus = (unsigned long long *)arena_alloc(A, 8ull * ((k + LB_TILE - 1) / LB_TILE), &ok);
            ws.lbCounter = (int32_t *)arena_alloc(A, 4, &ok);
            if (!ok) I->status = RR_ERR_WORKSPACE;
            s_ok = live(I);
        }
        __syncthreads();
        if (!s_ok) return;
        for (int64_t t = threadIdx.x; t < (k + LB_TILE - 1) / LB_TILE; t += blockDim.x) ws.lbStatus[t] = 0ull;
        if (threadIdx.x == 0) { *ws.lbCounter = 0; ws.ready0[k] = 0; }
        for (int c = threadIdx.x; c <= n; c += blockDim.x) { ws.colOff[c] = 0; ws.colCur[c] = 0; }
        for (int r = threadIdx.x; r <= m; r += blockDim.x) { ws.rowOff[r] = 0; ws.rowCur[r] = 0; }
        return;
    }
    if (threadIdx.x == 0) s_bad = 0;
    __syncthreads();
    long long P = 0, steps = 0;
    for (int64_t b = threadIdx.x; b < k; b += blockDim.x) {
        const rr_move p = load_move(&I->moves[b]);
        if (p.src_row < 0 || p.src_row >= m || p.dst_row < 0 || p.dst_row >= m || p.src_col < 0 ||
            p.src_col >= n || p.dst_col < 0 || p.dst_col >= n || (p.src_row == p.dst_row && p.src_col == p.dst_col))
            s_bad = 1;
        const int len = iabs(p.dst_col - p.src_col) + iabs(p.dst_row - p.src_row);
        steps += len; P += len + 1;
    }
    for (int o = 16; o; o >>= 1) {
        P += __shfl_xor_sync(FULL, P, o);
        steps += __shfl_xor_sync(FULL, steps, o);
    }
    if ((threadIdx.x & 31) == 0) { s_tmp[threadIdx.x >> 5] = P; s_tmp[16 + (threadIdx.x >> 5)] = steps; }
    __syncthreads();
    if (threadIdx.x == 0) {
        long long tp = 0, ts = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) { tp += s_tmp[w]; ts += s_tmp[16 + w]; }
        I->n_steps = ts;
        I->n_members = ts;
        if (s_bad) { I->status = RR_ERR_ARG; }
        else if (tp > 0x7fffffffLL) { I->status = RR_ERR_ARG; }
        else if (ts > I->cap_members || (ts > 0 && (!I->members || !I->ops))) {
            I->status = RR_ERR_CAPACITY;
            I->n_ops = ts;                      // upper bound
        } else {
            bool ok = true;
            const unsigned long long cells = (unsigned long long)m * n;
            ws.P = tp;
            ws.pairOff = (int32_t *)arena_alloc(A, 4ull * (k + 1), &ok);
            ws.nextAt = (int32_t *)arena_alloc(A, 4ull * (tp + 1), &ok);
            ws.colOff = (int32_t *)arena_alloc(A, 4ull * (n + 1), &ok);
            ws.colCur = (int32_t *)arena_alloc(A, 4ull * (n + 1), &ok);
            ws.colList = (int32_t *)arena_alloc(A, 4ull * (k + 1), &ok);
            ws.rowOff = (int32_t *)arena_alloc(A, 4ull * (m + 1), &ok);
            ws.rowCur = (int32_t *)arena_alloc(A, 4ull * (m + 1), &ok);
            ws.rowList = (int32_t *)arena_alloc(A, 4ull * (k + 1), &ok);
            ws.firstH = (int32_t *)arena_alloc(A, 4ull * cells, &ok);
            ws.multiMove = (int2 *)arena_alloc(A, 8ull * (k + 1), &ok);
            ws.indeg = (int32_t *)arena_alloc(A, 4ull * (k + 1), &ok);
            ws.rec = (int4 *)arena_alloc(A, 32ull * (k + 1), &ok);   // record, successors: one 32 B sector
            ws.ready0 = (int32_t *)arena_alloc(A, 4ull * (k + 1) + 16, &ok);
            ws.state = (int2 *)arena_alloc(A, sim_wide_bytes(k), &ok);
            ws.multi = ws.colList;               // both lists are free again once they have been swept
            ws.multiNo = ws.rowList;
            ws.nmulti = 0;
            // a path has at most as many successors as vertices: they
            // are stored at the path's vertex offset, so no count pass or scan
            ws.succ = (int32_t *)arena_alloc(A, 4ull * (tp + 1), &ok);
            ws.lbStatus = nullptr;
            ws.lbCounter = nullptr;
            if (!ok) I->status = RR_ERR_WORKSPACE;
        }
    }
    __syncthreads();
    if (!live(I)) return;
    // pairOff = exclusive scan of (len + 1); zero the counters
    for (int64_t b = threadIdx.x; b < k; b += blockDim.x) {
        const rr_move p = load_move(&I->moves[b]);
        ws.pairOff[b] = iabs(p.dst_col - p.src_col) + iabs(p.dst_row - p.src_row) + 1;
        ws.indeg[b] = 0;
    }
    if (threadIdx.x == 0) ws.ready0[k] = 0;      // count of initially ready moves
    for (int c = threadIdx.x; c <= n; c += blockDim.x) { ws.colOff[c] = 0; ws.colCur[c] = 0; }
    for (int r = threadIdx.x; r <= m; r += blockDim.x) { ws.rowOff[r] = 0; ws.rowCur[r] = 0; }
    __syncthreads();
    const long long tot = block_exclusive_scan(ws.pairOff, (int)k, s_tmp);
    if (threadIdx.x == 0) ws.pairOff[k] = (int32_t)tot;
}

// Path-vertex offsets of a large move list: pairOff[b] = sum over a < b of
// (path length + 1), by a single pass of decoupled look-back (Merrill and
// Garland, "Single-pass parallel prefix scan with decoupled look-back",
// 2016). Blocks take tiles of LB_TILE moves in order from the instance's
// counter (so every tile a block waits on is held by a running block); a
// tile publishes its aggregate at once and, once its exclusive prefix is
// known from the preceding tiles' words, its inclusive prefix. Status word:
// flag in the top two bits (0 not ready, 1 aggregate, 2 inclusive prefix),
// value in the low 62. Waits are bounded: a block that sees no progress for
// LB_SPIN_LIMIT polls sets RR_ERR_TIMEOUT and stops. The same pass checks
// every move, clears the in-degrees, and the block of the last tile, which
// learns the total, counts the elementary steps, checks the output room and
// allocates the vertex-sized arrays.
constexpr unsigned long long LB_AGG = 1ull << 62, LB_INCL = 2ull << 62, LB_VAL = (1ull << 62) - 1;
constexpr int LB_SPIN_LIMIT = 1 << 22;

__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release_u64(unsigned long long *p, unsigned long long v)
{
    asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ inline void s_pairoff_lookback(const Blk B, rr_instance *inst, JobWS *wsv, int count, Arena A)
{
    __shared__ long long s_warp[LB_THREADS / 32];
    __shared__ long long s_excl;
    __shared__ int s_tile, s_stop;
    const int q = B.y;
    if (q >= count) return;
    rr_instance *I = &inst[q];
    if (!live(I)) return;
    JobWS &ws = wsv[q];
    if (!ws.lbStatus) return;
    const int64_t k = I->n_moves;
    const int ntile = (int)((k + LB_TILE - 1) / LB_TILE);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    for (;;) {
        if (tid == 0) { s_tile = atomicAdd(ws.lbCounter, 1); s_stop = 0; }
        __syncthreads();
        const int tile = s_tile;
        if (tile >= ntile) break;
        // this thread's LB_ITEMS consecutive moves
        const int64_t b0 = (int64_t)tile * LB_TILE + (int64_t)tid * LB_ITEMS;
        int v[LB_ITEMS];
        long long sum = 0;
        bool bad = false;
        const int m = I->m, n = I->n;
#pragma unroll
        for (int u = 0; u < LB_ITEMS; ++u) {
            const int64_t b = b0 + u;
            v[u] = 0;
            if (b < k) {
                const rr_move p = load_move(&I->moves[b]);
                bad |= p.src_row < 0 || p.src_row >= m || p.dst_row < 0 || p.dst_row >= m || p.src_col < 0 ||
                       p.src_col >= n || p.dst_col < 0 || p.dst_col >= n ||
                       (p.src_row == p.dst_row && p.src_col == p.dst_col);
                v[u] = iabs(p.dst_col - p.src_col) + iabs(p.dst_row - p.src_row) + 1;
                ws.indeg[b] = 0;
            }
            sum += v[u];
        }
        if (bad) set_status(I, RR_ERR_ARG);
        // block scan of the thread sums
        long long incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long t = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) s_warp[wid] = incl;
        __syncthreads();
        if (wid == 0) {
            const long long w = lane < LB_THREADS / 32 ? s_warp[lane] : 0;
            long long wi = w;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const long long t = __shfl_up_sync(FULL, wi, o);
                if (lane >= o) wi += t;
            }
            if (lane < LB_THREADS / 32) s_warp[lane] = wi - w;
            const long long agg = __shfl_sync(FULL, wi, 31);
            if (lane == 0) {
                unsigned long long *st = ws.lbStatus;
                long long excl = 0;
                if (tile == 0) {
                    st_release_u64(&st[0], LB_INCL | (unsigned long long)agg);
                } else {
                    st_release_u64(&st[tile], LB_AGG | (unsigned long long)agg);
                    int j = tile - 1, spins = 0;
                    while (j >= 0) {
                        const unsigned long long w2 = ld_acquire_u64(&st[j]);
                        const unsigned long long f = w2 & ~LB_VAL;
                        if (f == 0ull) {
                            if (++spins > LB_SPIN_LIMIT) { s_stop = 1; break; }
                            __nanosleep(32);
                            continue;
                        }
                        spins = 0;
                        excl += (long long)(w2 & LB_VAL);
                        if (f == LB_INCL) break;
                        --j;
                    }
                    if (!s_stop) st_release_u64(&st[tile], LB_INCL | (unsigned long long)(excl + agg));
                }
                s_excl = excl;
                if (tile == ntile - 1 && !s_stop) {
                    // the total: elementary steps, the room they need, and
                    // the vertex-sized arrays (as the one-block set-up does)
                    const long long tp = excl + agg, ts = tp - k;
                    I->n_steps = ts;
                    I->n_members = ts;
                    if (tp > 0x7fffffffLL) {
                        set_status(I, RR_ERR_ARG);
                    } else if (ts > I->cap_members || (ts > 0 && (!I->members || !I->ops))) {
                        if (atomicCAS(&I->status, RR_OK, RR_ERR_CAPACITY) == RR_OK) I->n_ops = ts;
                    } else {
                        bool ok = true;
                        ws.P = tp;
                        ws.pairOff[k] = (int32_t)tp;
                        ws.nextAt = (int32_t *)arena_alloc(A, 4ull * (tp + 1), &ok);
                        ws.succ = (int32_t *)arena_alloc(A, 4ull * (tp + 1), &ok);
                        if (!ok) set_status(I, RR_ERR_WORKSPACE);
                    }
                }
            }
        }
        __syncthreads();
        if (s_stop) {
            if (tid == 0) set_status(I, RR_ERR_TIMEOUT);
            break;
        }
        long long run = s_excl + s_warp[wid] + incl - sum;
#pragma unroll
        for (int u = 0; u < LB_ITEMS; ++u) {
            const int64_t b = b0 + u;
            if (b < k) ws.pairOff[b] = (int32_t)run;
            run += v[u];
        }
        __syncthreads();
    }
}

constexpr int INTMAX = 0x7fffffff;

// Sort a[0..n) of int32 ascending with one warp: in registers up to 32, else
// by a bitonic network whose comparators all point up (each merge begins with
// a mirrored step), so that no padding is needed: in buf (cap words) when the
// list fits there, else in place.
__device__ inline void warp_sort32(int32_t *a, int n, int32_t *buf, int cap)
{
    const int lane = threadIdx.x & 31;
    if (n <= 1) return;
    if (n <= 32) {
        int v = lane < n ? a[lane] : 0x7fffffff;
#pragma unroll
        for (int kk = 2; kk <= 32; kk <<= 1) {
#pragma unroll
            for (int jj = kk >> 1; jj > 0; jj >>= 1) {
                const int o = __shfl_xor_sync(FULL, v, jj);
                const bool up = (lane & kk) == 0, low = (lane & jj) == 0;
                v = (low == up) ? min(v, o) : max(v, o);
            }
        }
        if (lane < n) a[lane] = v;
        __syncwarp();
        return;
    }
    int32_t *t = n <= cap ? buf : a;
    if (t != a)
        for (int i = lane; i < n; i += 32) t[i] = a[i];
    __syncwarp();
    auto order = [&](int i, int j) {
        if (j > i && j < n) {
            const int x = t[i], y = t[j];
            if (x > y) { t[i] = y; t[j] = x; }
        }
    };
    for (int k = 2; (k >> 1) < n; k <<= 1) {
        for (int i = lane; i < n; i += 32) order(i, i ^ (k - 1));
        __syncwarp();
        for (int j = k >> 2; j > 0; j >>= 1) {
            for (int i = lane; i < n; i += 32) order(i, i ^ j);
            __syncwarp();
        }
    }
    if (t != a)
        for (int i = lane; i < n; i += 32) a[i] = t[i];
    __syncwarp();
}

// A pointer loaded from memory, known to be global: loads and stores through
// it need not tell shared memory apart.
template <class T> __device__ __forceinline__ T *as_global(T *p)
{
    __builtin_assume(__isGlobal(p));
    return p;
}

// ---------------------------------------------------------------- Gamma
// Vertex (r, c) is covered by the vertical parts of the moves ending in
// column c (the corner of an L-move included) and by the horizontal parts of
// the L-moves running along row r (their destination column excluded). Two
// sweeps in id order -- one per row over the L-moves on it, one per column
// over the moves ending there -- give each vertex's horizontal and vertical
// coverers as two id-ordered chains. In red-rec plans every vertical
// coverer precedes every horizontal one (a corridor only crosses a column
// after that column's moves were emitted), so the chains are concatenated;
// elsewhere (bird's corridors cross columns solved later) the column sweep
// merges the two chains of that vertex by id (a chain holds each move at
// most once, so a merge takes at most k steps; more is an invariant failure).

__device__ inline void s_gcount(const Blk B, rr_instance *inst, JobWS *wsv, int count)
{
    const int q = B.y;
    if (q >= count) return;
    const rr_instance *I = &inst[q];
    if (!live(I)) return;
    JobWS &ws = wsv[q];
    const int64_t k = I->n_moves;
    for (int64_t b = B.x * blockDim.x + threadIdx.x; b < k; b += (int64_t)B.gx * blockDim.x) {
        const rr_move p = load_move(&I->moves[b]);
        atomicAdd(&ws.colCur[p.dst_col], 1);
        if (p.src_col != p.dst_col) atomicAdd(&ws.rowCur[p.src_row], 1);
    }
}

__device__ inline void s_gscan(const Blk B, rr_instance *inst, JobWS *wsv, int count)
{
    const int q = B.x;
    if (q >= count) return;
    const rr_instance *I = &inst[q];
    if (!live(I)) return;
    JobWS &ws = wsv[q];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (wid > 1) return;
    // warp 0: columns, warp 1: rows
    const int len = wid == 0 ? I->n : I->m;
    int32_t *cnt = wid == 0 ? ws.colCur : ws.rowCur, *off = wid == 0 ? ws.colOff : ws.rowOff;
    int carry = 0;
    for (int base = 0; base < len; base += 32) {
        const int i = base + lane;
        const int v = i < len ? cnt[i] : 0;
        const int incl = warp_incl_scan(v);
        if (i < len) { off[i] = carry + incl - v; cnt[i] = carry + incl - v; }
        carry += __shfl_sync(FULL, incl, 31);
    }
    if (lane == 0) off[len] = carry;
}

__device__ inline void s_gfill(const Blk B, rr_instance *inst, JobWS *wsv, int count)
{
    const int q = B.y;
    if (q >= count) return;
    const rr_instance *I = &inst[q];
    if (!live(I)) return;
    JobWS &ws = wsv[q];
    const int64_t k = I->n_moves;
    for (int64_t b = B.x * blockDim.x + threadIdx.x; b < k; b += (int64_t)B.gx * blockDim.x) {
        const rr_move p = load_move(&I->moves[b]);
        ws.colList[atomicAdd(&ws.colCur[p.dst_col], 1)] = (int32_t)b;
        if (p.src_col != p.dst_col) ws.rowList[atomicAdd(&ws.rowCur[p.src_row], 1)] = (int32_t)b;
    }
}

// Order every column list and row list by id (one warp per list). Lists of
// red-rec plans are mostly ascending already, and hold no more moves than
// the line has traps; a longer list (any move list may be batched) does not
// fit the buffer and is sorted in place.
__device__ inline void s_gsort(const Blk B, rr_instance *inst, JobWS *wsv, int count, int bufLen)
{
    extern __shared__ int32_t sortbuf[];
    const int q = B.y;
    if (q >= count) return;
    const rr_instance *I = &inst[q];
    if (!live(I)) return;
    JobWS &ws = wsv[q];
    const int lane = threadIdx.x & 31;
    int32_t *buf = sortbuf + (threadIdx.x >> 5) * bufLen;
    const int nl = I->n + I->m;
    for (int l = B.x * (blockDim.x >> 5) + (threadIdx.x >> 5); l < nl; l += B.gx * (blockDim.x >> 5)) {
        const bool col = l < I->n;
        const int idx = col ? l : l - I->n;
        int32_t *a = col ? ws.colList + ws.colOff[idx] : ws.rowList + ws.rowOff[idx];
        const int len = col ? ws.colOff[idx + 1] - ws.colOff[idx] : ws.rowOff[idx + 1] - ws.rowOff[idx];
        bool sorted = true;
        for (int i = lane; i + 1 < len; i += 32) sorted &= a[i] < a[i + 1];
        if (__all_sync(FULL, sorted)) continue;
        warp_sort32(a, len, buf, bufLen);
    }
}

// Calls f(id, first line crossed, legs' length, +-1, offset of the leg's first
// vertex) for the moves list[e0 .. e1) in order, for their horizontal legs or
// their vertical ones (one warp). The moves are read 32 at a time, one per
// lane, so that the loads' latency is paid once for 32 of them (4096 mixed grids:
// columns 3.0 -> 1.4 ms, rows 0.57 -> 0.35).
template <class F>
__device__ __forceinline__ void sweep_line(const rr_instance *I, const JobWS &ws, const int32_t *list, int e0, int e1,
                                           bool horizontal, F f)
{
    const int lane = threadIdx.x & 31;
    for (int g = e0; g < e1; g += 32) {
        int b = 0, leg = 0, base = 0;
        if (g + lane < e1) {
            b = list[g + lane];
            const rr_move p = load_move(&I->moves[b]);
            base = ws.pairOff[b];
            const int dr = p.dst_row - p.src_row, dc = p.dst_col - p.src_col;
            if (horizontal) leg = p.src_col | iabs(dc) << 10 | (dc > 0 ? 1 << 20 : 0);
            else { leg = p.src_row | iabs(dr) << 10 | (dr > 0 ? 1 << 20 : 0); base += iabs(dc); }
        }
        for (int i = 0; i < min(32, e1 - g); ++i) {
            const int l = __shfl_sync(FULL, leg, i);
            f(__shfl_sync(FULL, b, i), l & 1023, l >> 10 & 1023, l >> 20 ? 1 : -1, __shfl_sync(FULL, base, i));
            __syncwarp();
        }
    }
}

// Row sweep: the L-moves along each row in id order; each vertex's
// consecutive horizontal coverers are linked, the first is recorded.
__device__ inline void s_gsweep_h(const Blk B, rr_instance *inst, JobWS *wsv, int count, int lineCap)
{
    extern __shared__ int32_t sweepbuf[];
    const int q = B.y;
    if (q >= count) return;
    const rr_instance *I = &inst[q];
    if (!live(I)) return;
    JobWS &ws = wsv[q];
    const int lane = threadIdx.x & 31;
    const int n = I->n, m = I->m;
    int32_t *lastPos = sweepbuf + (threadIdx.x >> 5) * lineCap;
    for (int r = B.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < m; r += B.gx * (blockDim.x >> 5)) {
        for (int c = lane; c < n; c += 32) { lastPos[c] = -1; ws.firstH[(size_t)r * n + c] = -1; }
        __syncwarp();
        sweep_line(I, ws, ws.rowList, ws.rowOff[r], ws.rowOff[r + 1], true, [&](int b, int from, int len, int step, int base) {
            for (int t = lane; t < len; t += 32) {      // the destination column is the corner
                const int c = from + t * step;
                const int prev = lastPos[c];
                if (prev >= 0) ws.nextAt[prev] = b;
                else ws.firstH[(size_t)r * n + c] = b;
                lastPos[c] = base + t;
            }
        });
        for (int c = lane; c < n; c += 32)
            if (lastPos[c] >= 0) ws.nextAt[lastPos[c]] = -1;
        __syncwarp();
    }
}


// Column sweep: the moves ending in each column in id order; consecutive
// vertical coverers are linked, the last one to the vertex's first
// horizontal coverer. Where a horizontal coverer precedes a vertical one (a
// bird corridor through a column solved later), the two id-ordered chains of
// that vertex are merged by id instead.
__device__ inline void s_gsweep_v(const Blk B, rr_instance *inst, JobWS *wsv, int count, int lineCap)
{
    extern __shared__ int32_t sweepbuf[];
    const int q = B.y;
    if (q >= count) return;
    rr_instance *I = &inst[q];
    if (!live(I)) return;
    JobWS &ws = wsv[q];
    const int lane = threadIdx.x & 31;
    const int n = I->n, m = I->m;
    const int64_t k = I->n_moves;
    int32_t *lastPos = sweepbuf + (threadIdx.x >> 5) * 3 * lineCap;
    int32_t *lastId = lastPos + lineCap;
    int32_t *firstId = lastId + lineCap;
    for (int c = B.x * (blockDim.x >> 5) + (threadIdx.x >> 5); c < n; c += B.gx * (blockDim.x >> 5)) {
        for (int r = lane; r < m; r += 32) lastPos[r] = -1;
        __syncwarp();
        sweep_line(I, ws, ws.colList, ws.colOff[c], ws.colOff[c + 1], false, [&](int b, int from, int len, int step, int base) {
            for (int t = lane; t <= len; t += 32) {     // t = 0 is the corner / the source
                const int r = from + t * step;
                const int prev = lastPos[r];
                if (prev >= 0) ws.nextAt[prev] = b;
                else firstId[r] = b;
                lastPos[r] = base + t;
                lastId[r] = b;
            }
        });
        bool bad = false;
        for (int r = lane; r < m; r += 32) {
            if (lastPos[r] < 0) continue;
            const int f = ws.firstH[(size_t)r * n + c];
            if (f < 0 || f > lastId[r]) {              // every vertical coverer first
                ws.nextAt[lastPos[r]] = f;
                continue;
            }
            // merge: take the smaller id of the two chain heads, link it
            // after the previous one, advance its chain
            // (a head's vertex and successor are loaded when it becomes the
            // head, long before they are needed if the other chain goes first)
            auto vertex = [&](int x, bool vert) {
                const rr_move p = load_move(&I->moves[x]);
                return ws.pairOff[x] + (vert ? iabs(p.dst_col - p.src_col) + iabs(r - p.src_row) : iabs(c - p.src_col));
            };
            auto after = [&](int e, bool vert) { return vert && e == lastPos[r] ? -1 : ws.nextAt[e]; };
            int v = firstId[r], h = f, prevEntry = -1;
            int ve = vertex(v, true), he = vertex(h, false);
            int vn = after(ve, true), hn = after(he, false);
            int64_t steps = 0;
            for (; (v >= 0 || h >= 0) && steps <= k; ++steps) {   // a chain holds each move at most once
                const bool takeV = h < 0 || (v >= 0 && v < h);
                if (prevEntry >= 0) ws.nextAt[prevEntry] = takeV ? v : h;
                prevEntry = takeV ? ve : he;
                const int x = takeV ? vn : hn;
                int xe = -1, xn = -1;
                if (x >= 0) { xe = vertex(x, takeV); xn = after(xe, takeV); }
                if (takeV) { v = x; ve = xe; vn = xn; }
                else { h = x; he = xe; hn = xn; }
            }
            if (prevEntry >= 0) ws.nextAt[prevEntry] = -1;
            bad |= steps > k;
        }
        if (__any_sync(FULL, bad) && lane == 0) set_status(I, RR_ERR_INTERNAL);
        __syncwarp();
    }
}

// Successors of one path, written to out[0..) (each also counted in the
// successor's in-degree); returns their number, at most one per vertex.
// Consecutive path vertices mostly share their next path, so most entries
// repeat the previous one; a corridor that crosses many columns meets the next
// corridor again between them, which the four most recent successors catch. A
// successor that comes again later than that is counted twice, here and in its
// in-degree alike. (Comparing with all earlier ones, read back from out, took
// longest by far for the corridors of large grids: 1024 x 1024 1300 -> 229 us,
// 4096 mixed grids 2.1 -> 1.4 ms.) The path's entries
// are read 16 bytes at a time once aligned, the next 16 while these are
// compared.
__device__ inline int path_succ(const int32_t *seq, int len, int32_t *out, JobWS &ws)
{
    int cnt = 0;
    int32_t b0 = -1, b1 = -1, b2 = -1, b3 = -1;     // most recent first
    auto visit = [&](int32_t v) {
        if (v < 0 || v == b0) return;
        const bool again = v == b1 || v == b2 || v == b3;
        if (v != b1) {
            if (v != b2) b3 = b2;
            b2 = b1;
        }
        b1 = b0;
        b0 = v;
        if (again) return;
        out[cnt++] = v;
        atomicAdd(&ws.indeg[v], 1);              // (nothing waits for its answer)
    };
    int t = 0;
    const int head = min(len, (int)((4u - (unsigned)(((uintptr_t)seq >> 2) & 3u)) & 3u));
    for (; t < head; ++t) visit(seq[t]);
    int4 q = t + 4 <= len ? *reinterpret_cast<const int4 *>(seq + t) : make_int4(-1, -1, -1, -1);
    for (; t + 4 <= len; t += 4) {
        const int4 now = q;
        if (t + 8 <= len) q = *reinterpret_cast<const int4 *>(seq + t + 4);
        visit(now.x); visit(now.y); visit(now.z); visit(now.w);
    }
    for (; t < len; ++t) visit(seq[t]);
    return cnt;
}

// Successors of every path, written at the path's vertex offset,
// their count, and the in-degree of every successor.
__device__ inline void s_bsucc(const Blk B, rr_instance *inst, JobWS *wsv, int count)
{
    const int q = B.y;
    if (q >= count) return;
    const rr_instance *I = &inst[q];
    if (!live(I)) return;
    JobWS &ws = wsv[q];
    const int64_t k = I->n_moves;
    for (int64_t b = B.x * blockDim.x + threadIdx.x; b < k; b += (int64_t)B.gx * blockDim.x) {
        const int lo = ws.pairOff[b], hi = ws.pairOff[b + 1];
        ws.rec[2 * b].z = path_succ(ws.nextAt + lo, hi - lo, ws.succ + lo, ws);   // until the records are made
    }
}

// A number for every move with several predecessors, in no order.
__device__ inline void s_bnum(const Blk B, rr_instance *inst, JobWS *wsv, int count)
{
    const int q = B.y;
    if (q >= count) return;
    const rr_instance *I = &inst[q];
    if (!live(I)) return;
    JobWS &ws = wsv[q];
    const int64_t k = I->n_moves;
    const int lane = threadIdx.x & 31;
    for (int64_t b0 = B.x * blockDim.x + threadIdx.x - lane; b0 < k; b0 += (int64_t)B.gx * blockDim.x) {
        const int64_t b = b0 + lane;
        const bool several = b < k && ws.indeg[b] > 1;
        const unsigned bal = __ballot_sync(FULL, several);
        if (!bal) continue;
        int at = 0;
        if (lane == 0) at = atomicAdd(&ws.nmulti, __popc(bal));
        const int x = __shfl_sync(FULL, at, 0) + __popc(bal & ((1u << lane) - 1u));
        if (several) { ws.multiMove[x].x = (int)b; ws.multiNo[b] = x; }
    }
}

// Per-move records for the simulation: geometry, successor count and the
// first four successors (the flagged id of a successor without other
// predecessors, else the number of its counter); later successors are
// replaced in place. The in-degrees of the numbered moves start the
// simulation's counters; moves without predecessors are listed as ready.
__device__ inline void s_brec(const Blk B, rr_instance *inst, JobWS *wsv, int count)
{
    const int q = B.y;
    if (q >= count) return;
    const rr_instance *I = &inst[q];
    if (!live(I)) return;
    JobWS &ws = wsv[q];
    const int64_t k = I->n_moves;
    for (int64_t b = B.x * blockDim.x + threadIdx.x; b < k; b += (int64_t)B.gx * blockDim.x) {
        const rr_move p = load_move(&I->moves[b]);
        const int lo = ws.pairOff[b], hi = lo + ws.rec[2 * b].z;
        int v[4] = {-1, -1, -1, -1}, next = 0;
        for (int e = lo; e < hi; ++e) {
            const int32_t sId = ws.succ[e];
            const int32_t f = ws.indeg[sId] == 1 ? sId | SUCC_SINGLE : ws.multiNo[sId];
            if (e - lo < 4) v[e - lo] = f; else ws.succ[e] = f;
            if (sId == b + 1 && e - lo < 4) next = e - lo + 1;
        }
        const int4 r = move_rec(p, hi - lo, lo + 4, hi - lo == 1 && v[0] == (int)(SUCC_SINGLE | (b + 1)), next);
        ws.rec[2 * b] = r;
        ws.rec[2 * b + 1] = make_int4(v[0], v[1], v[2], v[3]);
        const int in = ws.indeg[b];
        if (in > 1) {
            const int x = ws.multiNo[b];
            ws.multi[x] = in | (r.y & 8191) << MULTI_BITS;
            ws.multiMove[x].y = r.x;
        }
        if (in == 0) ws.ready0[atomicAdd(&ws.ready0[k], 1)] = (int32_t)b;
    }
}

// Instance order by side, largest first: a counting sort on max(m, n)
// (one block; positions within a side follow the atomics, which does not
// matter: instances are independent). perm[i] is the instance at position i.
__device__ inline void s_order(const Blk B, const rr_instance *inst, int count, int *perm)
{
    __shared__ int hist[RR_MAX_SIDE + 2];
    for (int i = threadIdx.x; i < RR_MAX_SIDE + 2; i += blockDim.x) hist[i] = 0;
    __syncthreads();
    auto key = [&](int q) { return RR_MAX_SIDE + 1 - min(max(max(inst[q].m, inst[q].n), 0), RR_MAX_SIDE + 1); };
    for (int q = threadIdx.x; q < count; q += blockDim.x) atomicAdd(&hist[key(q)], 1);
    __syncthreads();
    if (threadIdx.x < 32) {              // exclusive scan, one warp
        int carry = 0;
        for (int b = 0; b < RR_MAX_SIDE + 2; b += 32) {
            const int i = b + threadIdx.x;
            const int v = i < RR_MAX_SIDE + 2 ? hist[i] : 0;
            const int inc = warp_incl_scan(v);
            if (i < RR_MAX_SIDE + 2) hist[i] = carry + inc - v;
            carry += __shfl_sync(FULL, inc, 31);
        }
    }
    __syncthreads();
    for (int q = threadIdx.x; q < count; q += blockDim.x) perm[atomicAdd(&hist[key(q)], 1)] = q;
}

// Descriptor copy in that order (one 128-byte descriptor per block).
__device__ inline void s_gather(const Blk B, const rr_instance *inst, const int *perm, rr_instance *pinst)
{
    const int32_t *src = (const int32_t *)&inst[perm[B.x]];
    int32_t *dst = (int32_t *)&pinst[B.x];
    dst[threadIdx.x] = src[threadIdx.x];
}

// Per-instance outputs back to the caller's descriptors.
__device__ inline void s_scatter(const Blk B, rr_instance *inst, const int *perm, const rr_instance *pinst, int count)
{
    for (int i = B.x * blockDim.x + threadIdx.x; i < count; i += B.gx * blockDim.x) {
        const rr_instance *p = &pinst[i];
        rr_instance *o = &inst[perm[i]];
        o->n_moves = p->n_moves;
        o->n_steps = p->n_steps;
        o->n_ops = p->n_ops;
        o->n_members = p->n_members;
        o->status = p->status;
    }
}

// Instances grouped by size class (largest side <= classSide[c]) so that each
// class's simulation launch gets shared memory sized for its own grids.
__device__ inline void s_classify(const Blk B, rr_instance *inst, int count, int nclass, int max_side, int *classCount,
                           int *classList)
{
    for (int q = B.x * blockDim.x + threadIdx.x; q < count; q += B.gx * blockDim.x) {
        const rr_instance *I = &inst[q];
        if (!live(I)) continue;
        const int side = max(I->m, I->n);
        int c = 0;
        while (c < nclass - 1 && side > class_side(max_side, c, nclass)) ++c;
        classList[c * count + atomicAdd(&classCount[c], 1)] = q;
    }
}

// ---------------------------------------------------------- simulation
//
// Alg. 4 with the local constraint set of Sec. IV, as an event-driven
// simulation: one block per instance; one warp simulates and logs, others
// write the batches.
//
// The lowest-id unfinished move is always ready (nothing earlier is
// unfinished), so it is always the first member ("leader") of the batch. With
// the leader's token at (r, c) moving in direction d, the other members are
// the ready moves stepping in direction d whose tokens lie on row r (set A)
// or on column c (set B): the one of A and B holding the smaller id wins,
// because pairwise row-or-column sharing with three or more tokens forces
// them onto one line. While the members advance together the batch can only
// change when the leg of one of them ends, or when the leader reaches a line
// across its way that holds a waiting ready move of direction d. Between such
// events every batch is the same: a segment.
//
// What bounds it: one warp's chain of dependent instructions (segments follow
// one another strictly; a 256 x 256 grid has about 29 000, its batches 724
// 000). So the state is laid out to keep that chain short:
//  - Coordinates are directed: a move of direction d has a position `along`
//    its way, mirrored for the two negative directions so that it always
//    grows, and `across` it. The leader's line across the way (its row, for a
//    vertical direction) is the set of equal `along`, its line of motion the
//    set of equal `across`.
//  - Ready moves outside the batch ("statics") stand in one table per
//    direction, `along` and `across` in the halves of a word, holes marked.
//    Two 16-byte loads per lane cover 256 statics; one fused add-and-minimum
//    on 16-bit halves per static tells whether any stands on one of the
//    leader's two lines and how far the next line ahead is. There are no
//    lists to walk or to maintain: a move enters by two stores, its entry
//    taken from a stack by one atomic, so that lanes need no vote among them.
//  - The batch's other members advance by a common clock: a member keeps its
//    `along` minus the clock and the clock at which its leg ends, so a segment
//    that none of them ends does not touch them. They are kept in no order
//    (the writers sort), with the smallest id and the first end in registers.
//  - The leader lives in registers. When it finishes, the next leader is
//    nearly always the next id, released at that moment; its record has been
//    brought into L1 long before. Successive leaders that meet nothing on
//    their way are taken together (run_of_leaders).
//  - In-degrees of the moves with several predecessors are counted in shared
//    memory as far as they fit (a global atomic's answer takes about 700
//    cycles); their predecessors name the counter, not the move, so that a
//    count that does not reach zero touches nothing else. Moves with one
//    predecessor need no count.
//  - A segment is logged in 16 bytes plus its members' ids where these
//    changed, into memory that the conflict graph no longer needs. Other
//    warps turn the log into batches and members, 32 segments at a time, with
//    stores of consecutive words: three warps of the same block while the
//    simulation runs on (calls over few grids), or a kernel after it.
// One 256 x 256 grid: 63 ms with linked lists, sorted members, batches written
// by the simulating warp and in-degrees in global memory; 17 ms this way.

// ------------------------------------------------------------- the writers

// What a lane writes of a segment's batches: three words per batch
// (direction, first member, count), a warp's store covering 32 consecutive
// words, so that 32 batches take three stores, in which a lane's words are
// always the same field (f) of the same batch (q) of the 32.
struct OpLane {
    int f[3], q[3];
    __device__ __forceinline__ OpLane(int lane)
    {
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            q[j] = (lane + 32 * j) / 3;
            f[j] = (lane + 32 * j) % 3;
        }
    }
};
__device__ __forceinline__ void write_ops(int32_t *o, const OpLane &P, int lane, unsigned mem0, int kseg, int ns, int d)
{
    int v[3], by[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        by[j] = P.f[j] == 1 ? ns : 0;
        v[j] = (P.f[j] == 0 ? d : P.f[j] == 1 ? (int)mem0 : ns) + by[j] * P.q[j];
    }
    for (int w = lane; w - lane < 3 * kseg; w += 96) {
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            if (w + 32 * j < 3 * kseg) o[w + 32 * j] = v[j];
            v[j] += 32 * by[j];
        }
    }
}

// The room that a capacity gives: none if it is negative.
__device__ __forceinline__ unsigned long long room_of(int64_t cap) { return cap > 0 ? (unsigned long long)cap : 0ull; }

// A segment's kseg batches of ns moves at batch op0 and member mem0: the
// leader L (the smallest id) and the ns - 1 moves of list[], in no order.
// One warp; buf holds the next power of two of ns words. Batches are written
// as consecutive words (three per batch), members likewise.
__device__ inline void write_segment(rr_op *ops, int32_t *mem, const OpLane &P, unsigned op0, unsigned mem0, int kseg,
                                     int ns, int d, int L, const int32_t *list, int32_t *buf)
{
    const int lane = threadIdx.x & 31;
    write_ops((int32_t *)(ops + op0), P, lane, mem0, kseg, ns, d);
    int32_t *mp = mem + mem0;
    const int total = kseg * ns;
    if (ns == 1) {
        for (int i = lane; i - lane < total; i += 32)
            if (i < total) mp[i] = L;
        return;
    }
    // lane's place in the cycle of ns members, and what 32 places on means
    const float inv = __frcp_rn((float)ns);
    auto mod = [&](int a) {
        int r = a - __float2int_rz((float)a * inv) * ns;
        if (r < 0) r += ns;
        if (r >= ns) r -= ns;
        return r;
    };
    int u = mod(lane);
    const int step = mod(32);
    if (ns <= 32) {
        int v = lane == 0 ? L : lane < ns ? list[lane - 1] : INTMAX;
        if (ns > 2) {              // sort: every lane counts the smaller ones
            int r = 0;
            for (int j = 1; j < ns; ++j) r += __shfl_sync(FULL, v, j) < v;
            if (lane > 0) ++r;     // the leader is the smallest
            if (lane < ns) buf[r] = v;
            __syncwarp();
            v = lane < ns ? buf[lane] : 0;
        }
        for (int i0 = 0; i0 < total; i0 += 32) {
            const int x = __shfl_sync(FULL, v, u);
            if (i0 + lane < total) mp[i0 + lane] = x;
            u += step;
            if (u >= ns) u -= ns;
        }
    } else {
        for (int i = lane; i < ns; i += 32) buf[i] = i == 0 ? L : list[i - 1];
        __syncwarp();
        warp_sort32(buf, ns, buf, ns);
        for (int i = lane; i < total; i += 32) {
            mp[i] = buf[u];
            u += step;
            if (u >= ns) u -= ns;
        }
    }
    __syncwarp();
}

constexpr int SIM_POLLS = 1 << 22;      // a writer's polls without progress of the log before it gives up

// Header of a logged segment: its first batch and first member, where its
// members' ids lie, and the leader (30 bits) with the direction. Lengths
// follow from the next header.
__device__ __forceinline__ void write_chunk(const int32_t *log, int s0, int cnt, unsigned long long cap_ops,
                                            unsigned long long cap_mem, rr_op *ops, int32_t *mem, const OpLane &P,
                                            int32_t *buf)
{
    const int lane = threadIdx.x & 31;
    const uint4 *hdr = (const uint4 *)log;
    uint4 h = make_uint4(0u, 0u, 0u, 0u);
    int kseg = 0, ns = 0;
    if (lane < cnt) {
        h = hdr[s0 + lane];
        const uint2 nx = *(const uint2 *)&hdr[s0 + lane + 1];
        kseg = (int)(nx.x - h.x);
        ns = (int)((nx.y - h.y) / (unsigned)max(kseg, 1));
        // a batch list that does not fit ends as RR_ERR_CAPACITY: nothing of it is written
        if (nx.x > cap_ops || nx.y > cap_mem) kseg = 0;
    }
    for (int j = 0; j < cnt; ++j) {
        const int kj = __shfl_sync(FULL, kseg, j), nj = __shfl_sync(FULL, ns, j);
        const unsigned op0 = __shfl_sync(FULL, h.x, j), mem0 = __shfl_sync(FULL, h.y, j);
        const unsigned lo = __shfl_sync(FULL, h.z, j), l = __shfl_sync(FULL, h.w, j);
        if (kj > 0)
            write_segment(ops, mem, P, op0, mem0, kj, nj, (int)(l >> 30), (int)(l & 0x3fffffffu), log + lo, buf);
    }
}

// A warp of the simulation's block writes what is published of the log, 32
// segments at a time, until the log has ended and nothing is left.
__device__ inline void run_writers(SimCtl *C, rr_instance *I, const int32_t *log, int32_t *buf)
{
    const int lane = threadIdx.x & 31;
    const unsigned long long cap_ops = room_of(I->cap_ops), cap_mem = room_of(I->cap_members);
    rr_op *ops = as_global(I->ops);
    int32_t *mem = as_global(I->members);
    volatile int *pub = &C->pub, *fin = &C->fin;
    const OpLane P(lane);
    for (;;) {
        int s0 = 0;
        if (lane == 0) s0 = atomicAdd(&C->next, 32);
        s0 = __shfl_sync(FULL, s0, 0);
        int have = 0;
        for (int polls = 0;; ++polls) {
            const int f = *fin;
            __threadfence_block();
            have = *pub;
            if (__all_sync(FULL, have >= s0 + 32 || f)) break;
            if (polls > SIM_POLLS) { if (lane == 0) set_status(I, RR_ERR_TIMEOUT); return; }
            __nanosleep(2000);
        }
        have = __shfl_sync(FULL, have, 0);
        __threadfence_block();
        const int cnt = min(32, have - s0);
        if (cnt <= 0) return;
        write_chunk(log, s0, cnt, cap_ops, cap_mem, ops, mem, P, buf);
    }
}

// The logged segments of every instance, as far as its simulation ran without
// writers of its own: a warp per 32 segments.
__device__ inline void s_write(const Blk B, rr_instance *I, const JobWS &ws, int32_t *buf)
{
    if (!live(I) || I->n_moves == 0) return;
    const int lane = threadIdx.x & 31;
    const OpLane P(lane);
    rr_op *ops = as_global(I->ops);
    int32_t *mem = as_global(I->members);
    const int32_t *log = as_global(ws.nextAt);
    const unsigned long long cap_ops = room_of(I->cap_ops), cap_mem = room_of(I->cap_members);
    for (int s0 = 32 * B.w; s0 < ws.nseg; s0 += 32 * B.nw)
        write_chunk(log, s0, min(32, ws.nseg - s0), cap_ops, cap_mem, ops, mem, P, buf);
}

// ---------------------------------------------------------- the simulation

// Position words: `along` in the low half, `across` in the high one, both
// plus one, so that neither is zero; a hole of the table is all ones.
constexpr uint32_t HOLE = 0xffffffffu;

// The vertical leg after a horizontal one (direction d) that ended at p.
struct Leg { int d; uint32_t pos; int rem; };
__device__ __forceinline__ Leg second_leg(int d, uint32_t p, int dstRow)
{
    const int row = (int)(p >> 16) - 1, al = (int)(p & 0xffffu);
    Leg g;
    g.d = dstRow > row ? 1 : 0;
    g.pos = dir_pos(g.d, row, d == 2 ? MIRROR - 1 - al : al - 1);
    g.rem = iabs(dstRow - row);
    return g;
}

// Which of eight position words match w in the halves of `half`.
__device__ __forceinline__ unsigned match8(uint4 a, uint4 b, uint32_t w, uint32_t half)
{
    const uint32_t x[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    unsigned m = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) m |= ((x[i] ^ w) & half) == 0u ? 1u << i : 0u;
    return m;
}
// Minimum, half by half, of v and the eight words plus w.
__device__ __forceinline__ uint32_t min8(uint4 a, uint4 b, uint32_t w, uint32_t v)
{
    v = __viaddmin_u16x2(a.x, w, v);
    v = __viaddmin_u16x2(a.y, w, v);
    v = __viaddmin_u16x2(a.z, w, v);
    v = __viaddmin_u16x2(a.w, w, v);
    v = __viaddmin_u16x2(b.x, w, v);
    v = __viaddmin_u16x2(b.y, w, v);
    v = __viaddmin_u16x2(b.z, w, v);
    v = __viaddmin_u16x2(b.w, w, v);
    return v;
}

// Memory operations of the lanes that `c` holds for, predicated rather than
// branched around: in one warp's serial code a branch and the point where its
// lanes meet again cost 15 to 20 cycles each, and the code below has little
// else between them.
#define RR_IF(instr) "{ .reg .pred q; setp.ne.u32 q, %0, 0; @q " instr " }"
__device__ __forceinline__ int sh_add_if(bool c, void *p, int v)
{
    int r = 0;
    asm volatile("{ .reg .pred q; setp.ne.u32 q, %1, 0; @q atom.shared.add.u32 %0, [%2], %3; }"
                 : "+r"(r) : "r"((unsigned)c), "r"(sh_addr(p)), "r"(v) : "memory");
    return r;
}
__device__ __forceinline__ int ld_u16_if(bool c, const uint16_t *p)
{
    unsigned short r = 0;
    asm volatile("{ .reg .pred q; setp.ne.u32 q, %1, 0; @q ld.shared.u16 %0, [%2]; }"
                 : "+h"(r) : "r"((unsigned)c), "r"(sh_addr(p)) : "memory");
    return r;
}
__device__ __forceinline__ void st_if(bool c, uint16_t *p, int v)
{
    asm volatile(RR_IF("st.shared.u16 [%1], %2;") ::"r"((unsigned)c), "r"(sh_addr(p)), "h"((unsigned short)v) : "memory");
}
__device__ __forceinline__ void st_if(bool c, void *p, uint32_t v)
{
    asm volatile(RR_IF("st.shared.u32 [%1], %2;") ::"r"((unsigned)c), "r"(sh_addr(p)), "r"(v) : "memory");
}
__device__ __forceinline__ void st_if(bool c, int2 *p, int x, int y)
{
    asm volatile(RR_IF("st.shared.v2.u32 [%1], {%2, %3};") ::"r"((unsigned)c), "r"(sh_addr(p)), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ int4 ldg_if(bool c, const int4 *p)
{
    int4 v = make_int4(0, 0, 0, 0);
    asm volatile("{ .reg .pred q; setp.ne.u32 q, %4, 0; @q ld.global.v4.u32 {%0, %1, %2, %3}, [%5]; }"
                 : "+r"(v.x), "+r"(v.y), "+r"(v.z), "+r"(v.w) : "r"((unsigned)c), "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ int2 ldg_if(bool c, const int2 *p)
{
    int2 v = make_int2(0, 0);
    asm volatile("{ .reg .pred q; setp.ne.u32 q, %2, 0; @q ld.global.v2.u32 {%0, %1}, [%3]; }"
                 : "+r"(v.x), "+r"(v.y) : "r"((unsigned)c), "l"(p) : "memory");
    return v;
}
// (not from L1: atomics change the word in L2)
__device__ __forceinline__ int ldg_volatile_if(bool c, const void *p)
{
    int v = 0;
    asm volatile("{ .reg .pred q; setp.ne.u32 q, %1, 0; @q ld.global.cg.u32 %0, [%2]; }"
                 : "+r"(v) : "r"((unsigned)c), "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ int ldg_if(bool c, const void *p)
{
    int v = 0;
    asm volatile("{ .reg .pred q; setp.ne.u32 q, %1, 0; @q ld.global.u32 %0, [%2]; }"
                 : "+r"(v) : "r"((unsigned)c), "l"(p) : "memory");
    return v;
}
#undef RR_IF

__device__ __forceinline__ void touch_rec_if(bool c, const int4 *rec, int id, uint32_t dump)
{
    touch_if(c, rec + 2 * (size_t)id, dump);
}

// The largest of the lanes' values (usually all the same): a value that the
// compiler knows to be uniform, so that branches on it, and on what is
// computed from it, need no bookkeeping for lanes that might diverge.
__device__ __forceinline__ uint32_t uni(uint32_t v) { return __reduce_max_sync(FULL, v); }


// A segment written by the simulating warp itself, once the log is full, out of
// line: the loop around it stays smaller (389 x 501 39.6 -> 38.0 ms; where
// registers are scarcest, in the small tables' kernel, inlining is better: 4096
// mixed grids 31 ms, 33 this way).
static __device__ __noinline__ void write_call(rr_instance *I, unsigned op0, unsigned mem0, int kseg, int ns, int d, int L,
                                               const int32_t *list, int32_t *buf)
{
    write_segment(as_global(I->ops), as_global(I->members), OpLane(lane_id()), op0, mem0, kseg, ns, d, L, list, buf);
}

constexpr int RUN = 32;     // leaders of a run at most: one per lane

// Segments that the log has room for: a header each, one after them, a list
// of ids each, and the headers of one run.
__device__ __forceinline__ int log_room(unsigned nseg, unsigned idTop, int lineCap)
{
    return ((int)idTop - 4 * ((int)nseg + 2 + 2 * RUN)) / (4 + lineCap);
}

// A block's shared memory (sim_smem_bytes), the tables apart.
struct SimLayout {
    int MC;                   // room of the members
    int2 *mie;
    uint32_t *mpos;
    SimCtl *C;
    int32_t *bufs, *ids;      // a sort buffer per warp, a list of ids
    int32_t *dump;            // 16 bytes that nothing reads
    unsigned *cnt;
    __device__ __forceinline__ SimLayout(char *smem, int side)
    {
        MC = (side + 7) & ~7;
        mie = (int2 *)(smem + 14 * 4 * sim_cap(side));
        mpos = (uint32_t *)(mie + MC);
        C = (SimCtl *)(mpos + MC);
        bufs = (int32_t *)(C + 1);
        ids = bufs + sim_pow2(side) * (int)(blockDim.x >> 5);
        dump = ids + MC;
        cnt = (unsigned *)(dump + 4);
    }
};

// A run: successive leaders, each alone in its batches, are taken
// together. Lane i looks at the i-th next id (lane 0 at the leader), its
// horizontal leg if it has one, and its vertical leg. The run goes on
// while every vertical leg runs the same way down the same column, no
// static stands on or ahead of either leg's line of motion or on a line
// that the leg reaches, the only move that a leader makes ready is the
// next id, and no in-degree counter of a successor runs out. Nothing else
// changes meanwhile, so the batches are known at once: the legs, one
// after another. Deep in a receiver's unit nearly all moves are of this
// kind: on a 256 x 256 grid 900 runs take 10 700 of 14 400 leaders (the
// simulation 22.4 -> 17.1 ms). The leader L has rem steps of its leg left at lpos in
// direction d. Returns 0 or the leaders taken, their legs (each logged) and
// their steps, in 6, 7 and 17 bits. Not inlined: its registers would crowd
// those of the loop that calls it.
template <int MODE>
static __device__ __noinline__ int run_of_leaders(rr_instance *I, JobWS *ws, char *smem, int side, int counters, int L, int d,
                                                  int rem, uint32_t lpos, int clk, unsigned nmem, unsigned nseg,
                                                  unsigned list, bool logging)
{
    const SimLayout Y(smem, side);
    const int lane = lane_id(), k = (int)I->n_moves, cap = sim_cap(side), groups = cap >> 3;
    const int ncnt = min(counters, ws->nmulti);
    const bool allShared = counters >= ws->nmulti;
    const uint32_t *pos = (const uint32_t *)smem;
    const int4 *rec = as_global(ws->rec);
    int32_t *multi = as_global(ws->multi), *log = as_global(ws->nextAt);
    const int2 *multiMove = as_global(ws->multiMove);
    SimCtl *C = Y.C;
    unsigned *cnt = Y.cnt;
    int32_t *ids = Y.ids, *buf = Y.bufs;
    const uint32_t dump = sh_addr(Y.dump);
    const int id = min(L + lane, k);
    const int4 r = rec[2 * (size_t)id], s = rec[2 * (size_t)id + 1];
    int d1 = r.y & 3, len = r.y >> 2 & 2047;
    uint32_t p1 = (uint32_t)r.x;
    if (lane == 0) { d1 = d; len = rem; p1 = lpos; }
    const bool hor = d1 >= 2;
    const Leg g = second_leg(d1, p1 + (uint32_t)len, r.y >> 13 & 1023);
    const int hl = hor ? len : 0, vd = hor ? g.d : d1, vl = hor ? g.rem : len;
    const uint32_t vp = hor ? g.pos : p1;
    const int rd = __shfl_sync(FULL, vd, 0);
    const uint32_t rc = __shfl_sync(FULL, vp >> 16, 0);
    // successors: the next id (without another predecessor, or the last
    // one it waits for), and counters that stay above zero
    const int32_t sv[4] = {s.x, s.y, s.z, s.w};
    const int next = (r.y >> 24 & 7) - 1;
    bool link = false, bad = L + lane >= k || r.z > 4 || vl == 0 || vd != rd || (vp >> 16) != rc;
    bool inS[4], inG[4];
    int left_[4];
    #pragma unroll
    for (int e = 0; e < 4; ++e) {
        const bool v = e < r.z && !bad, one = (sv[e] & SUCC_SINGLE) != 0;
        inS[e] = v && !one && sv[e] < ncnt;
        inG[e] = v && !one && sv[e] >= ncnt;
        link |= v && one && e == next;
    }
    #pragma unroll
    for (int e = 0; e < 4; ++e) {
        bad |= e < r.z && (sv[e] & SUCC_SINGLE) && e != next;
        left_[e] = ld_u16_if(inS[e], (const uint16_t *)cnt + (inS[e] ? sv[e] : 0));
    }
    if (!allShared)
    #pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int c = ldg_volatile_if(inG[e], multi + (inG[e] ? sv[e] : 0)) & MULTI_COUNT;
            left_[e] = inG[e] ? c : left_[e];
        }
    unsigned few = 0;       // entries whose counter will be at one
    #pragma unroll
    for (int e = 0; e < 4; ++e) {
        const bool m = inS[e] || inG[e], last = m && left_[e] == 1;
        link |= last && e == next;
        bad |= last && e != next;
        few |= m && left_[e] == 2 ? 1u << e : 0u;
        inS[e] = inS[e] && !last;          // (nobody else waits on a counter that has run out)
        inG[e] = inG[e] && !last;
    }
    const unsigned okb = __ballot_sync(FULL, !bad && link);
    int n = okb == FULL ? 32 : __ffs(~okb) - 1;
    if (n == 0) return 0;
    // horizontal legs against the few statics of the horizontal directions
    if (__any_sync(FULL, hl > 0))
        for (int q = 2; q < 4; ++q) {
            if (C->nfree[q] == cap) continue;
            bool hit = false;
            for (int g0 = 0; g0 < groups; g0 += 32) {
                const int e0 = q * cap + 8 * min(g0 + lane, groups - 1);
                const uint4 a = *(const uint4 *)(pos + e0), b = *(const uint4 *)(pos + e0 + 4);
                const uint32_t all = a.x & a.y & a.z & a.w & b.x & b.y & b.z & b.w;
                // (a hole is no hit: it lies far ahead, on no row)
                for (unsigned m = __ballot_sync(FULL, all != HOLE); m; m &= m - 1) {
                    const int src = 31 - __clz(m & (0u - m));
                    const uint32_t x[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    #pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const uint32_t w = __shfl_sync(FULL, x[u], src);
                        hit |= ((w - p1) & 0xffffu) < (unsigned)hl || (w >> 16) == (p1 >> 16);
                    }
                }
            }
            const unsigned hb = __ballot_sync(FULL, hit && d1 == q);
            if (hb) n = min(n, __ffs(hb) - 1);
        }
    // vertical legs against the statics of their direction, four at a time
    const int vtb = rd * cap;
    for (int i = 0; i < n; i += 4) {
        uint32_t w[4], v[4];
        int need[4];
    #pragma unroll
        for (int u = 0; u < 4; ++u) {
            w[u] = 0x10000u - __shfl_sync(FULL, vp, i + u);
            need[u] = __shfl_sync(FULL, vl, i + u);
            v[u] = HOLE;
        }
        for (int gg = 0; gg < groups; gg += 32) {
            const int e0 = vtb + 8 * min(gg + lane, groups - 1);
            const uint4 a = *(const uint4 *)(pos + e0), b = *(const uint4 *)(pos + e0 + 4);
    #pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = min8(a, b, w[u], v[u]);
        }
        int stop = n;
    #pragma unroll
        for (int u = 3; u >= 0; --u) {
            const int near = (int)__reduce_min_sync(FULL, v[u] < 0x10000u ? 0u : v[u] & 0xffffu);
            if (near < need[u]) stop = i + u;
        }
        if (stop < n) { n = stop; break; }
    }
    // count down; a counter that runs out after all (two leaders of the
    // run share it) ends the run before the last of them
    while (n > 0) {
        const bool in = lane < n;
        int gone = -1, old[4];
    #pragma unroll
        for (int e = 0; e < 4; ++e)
            old[e] = sh_add_if(in && inS[e], cnt + (inS[e] ? sv[e] >> 1 : 0), -(1 << ((sv[e] & 1) * 16)));
    #pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (in && inS[e] && (old[e] >> ((sv[e] & 1) * 16) & 0xffff) == 1) gone = sv[e];
            if (!allShared && in && inG[e] && (atomicSub(&multi[sv[e]], 1) & MULTI_COUNT) == 1) gone = sv[e];
        }
        const unsigned gb = __ballot_sync(FULL, gone >= 0);
        if (!gb) break;
        const int x = __shfl_sync(FULL, gone, __ffs(gb) - 1);
        bool has = false;
    #pragma unroll
        for (int e = 0; e < 4; ++e) {                        // take them back
            sh_add_if(in && inS[e], cnt + (inS[e] ? sv[e] >> 1 : 0), 1 << ((sv[e] & 1) * 16));
            if (!allShared && in && inG[e]) atomicAdd(&multi[sv[e]], 1);
            has |= in && (inS[e] || inG[e]) && sv[e] == x;
        }
        n = 31 - __clz(__ballot_sync(FULL, has));
        __syncwarp();
    }
    if (n == 0) return 0;
    if (__any_sync(FULL, lane < n && few != 0u)) {
    #pragma unroll
        for (int e = 0; e < 4; ++e) {
            const bool t = lane < n && (few >> e & 1u);
            touch_if(t, multiMove + (t ? sv[e] : 0), dump);
            touch_if(t, multi + (t ? sv[e] : 0), dump);
        }
    }
    // log the legs
    const int mine = lane < n ? (hl + vl) | ((hl > 0 ? 2 : 1) << 20) : 0;
    const int incl = warp_incl_scan(mine), tot = __shfl_sync(FULL, incl, 31);
    const int before = (incl - mine) & 0xfffff, steps = tot & 0xfffff, segs = tot >> 20;
    if (logging) {
        uint4 *h = (uint4 *)log + nseg + ((incl - mine) >> 20);
        if (lane < n) {
            if (hl > 0) *h++ = make_uint4((unsigned)(clk + before), nmem + (unsigned)before, list, (unsigned)id | (unsigned)d1 << 30);
            *h = make_uint4((unsigned)(clk + before + hl), nmem + (unsigned)(before + hl), list, (unsigned)id | (unsigned)vd << 30);
        }
    } else {
        for (int i = 0; i < n; ++i) {
            const int o = clk + __shfl_sync(FULL, before, i), m0 = (int)nmem + __shfl_sync(FULL, before, i);
            const int h1 = __shfl_sync(FULL, hl, i), v1 = __shfl_sync(FULL, vl, i), hd = __shfl_sync(FULL, d1, i);
            if ((unsigned long long)(o + h1 + v1) > room_of(I->cap_ops) ||
                (unsigned long long)(m0 + h1 + v1) > room_of(I->cap_members)) break;
            if (h1 > 0) write_segment(as_global(I->ops), as_global(I->members), OpLane(lane), (unsigned)o, (unsigned)m0, h1, 1, hd, L + i, ids, buf);
            write_segment(as_global(I->ops), as_global(I->members), OpLane(lane), (unsigned)(o + h1), (unsigned)(m0 + h1), v1, 1, rd, L + i, ids, buf);
        }
    }
    return n | segs << 6 | steps << 13;
}

// The log has ended and pub is final: the writers are done once they have
// written it, however long the simulation, writing by itself, still takes.
__device__ __forceinline__ void end_of_log(SimCtl *C)
{
    __threadfence_block();
    if (lane_id() == 0) *(volatile int *)&C->fin = 1;
}
// The end of a simulation: a header with the totals, everything published,
// the instance's counts. Returns its status.
__device__ __forceinline__ int sim_end(rr_instance *I, SimCtl *C, uint4 *hdr, unsigned nseg, bool logging, int clk,
                                       unsigned nmem, int err)
{
    const int lane = lane_id();
    touch_wait();
    __syncwarp();
    if (logging && lane == 0) hdr[nseg] = make_uint4((unsigned)clk, nmem, 0u, 0u);
    if (lane == 0) {
        I->n_ops = clk;
        I->n_members = nmem;
    }
    if (*(volatile int *)&C->full) err = RR_SIM_RETRY;
    if (!err && (long long)nmem != I->n_steps) err = RR_ERR_INTERNAL;
    if (!err && ((int64_t)clk > I->cap_ops || (int64_t)nmem > I->cap_members)) err = RR_ERR_CAPACITY;
    __syncwarp();
    __threadfence_block();
    if (lane == 0) *(volatile int *)&C->pub = (int)nseg;
    end_of_log(C);
    __syncwarp();
    return err;
}

// One simulation by one warp. SIM_SMALL: tables in shared memory, at most 256
// entries per direction (one load of every lane covers them); SIM_BIG: the
// same with more entries. Both end with RR_SIM_RETRY when an instance has
// more ready moves of a direction than entries (WideSim, below).
enum { SIM_SMALL, SIM_BIG };

template <int MODE>
struct Sim {
    uint32_t *pos;            // position words, a table of cap entries per direction
    int2 *ir;                 // id, steps left in the leg
    uint16_t *stk;            // free entries (numbers within the table)
    int cap;
    int2 *mie;                // members: id, clock at the end of the leg
    uint32_t *mpos;           // members: position word, `along` minus the clock
    SimCtl *C;
    const int4 *rec;
    const int32_t *succ;
    const int2 *multiMove;    // the moves that the counters belong to: id, position word
    int32_t *multi;           // in-degree counters in global memory (with their moves' first legs)
    unsigned *cnt;            // the first ncnt of them in shared memory, two per word
    int ncnt;
    bool allShared;           // all of them
    uint32_t dump;            // shared address for the touches
    char *smem;               // the block's shared memory, its side and counters
    int side, counters;

    // The moves of the lanes with c become statics.
    __device__ __forceinline__ void enter(bool c, int d, uint32_t p, int id, int rem)
    {
        const int o = sh_add_if(c, &C->nfree[d], -1) - 1;
        const bool none = c && o < 0, ok = c && o >= 0;
        st_if(none, &C->full, 1u);             // no room: the run will end with RR_SIM_RETRY
        sh_add_if(none, &C->nfree[d], 1);
        const int e = d * cap + ld_u16_if(ok, stk + d * cap + o);
        st_if(ok, pos + e, p);
        st_if(ok, ir + e, id, rem);
    }

    // A finished move of each lane with c hands one predecessor fewer to the
    // successor entry v: a move without other predecessors (flagged id) is
    // ready now, another counts down. The moves that become ready enter their
    // tables, except the next leader: true in its lane. (Every lane calls.)
    __device__ __forceinline__ bool release(bool c, int32_t v, int handId)
    {
        const bool single = c && (v & SUCC_SINGLE), multi_ = c && !(v & SUCC_SINGLE);
        const int x = v & SUCC_ID;
        const int sh = (x & 1) * 16;
        bool h = single && x == handId;
        const bool fresh = single && !h;
        int old = (sh_add_if(multi_ && x < ncnt, cnt + (x >> 1), -(1 << sh)) >> sh) & 0xffff;
        int2 r = ldg_if(fresh, (const int2 *)(rec + 2 * (size_t)x));       // (in flight during the vote)
        if (!allShared) {
            if (multi_ && x >= ncnt) old = atomicSub(&multi[x], 1) & MULTI_COUNT;
            __syncwarp();
        }
        const bool soon = multi_ && old == 2, last = multi_ && old == 1;
        touch_if(soon, multiMove + x, dump);         // next time it is ready
        touch_if(soon, multi + x, dump);
        if (__any_sync(FULL, fresh || last)) {
            const int2 mv = ldg_if(last, multiMove + x);
            const int y = ldg_if(last, (const void *)(multi + x)) >> MULTI_BITS;
            const int id = last ? mv.x : x;
            if (last) r = make_int2(mv.y, y);
            h |= last && id == handId;
            enter((fresh || last) && !h, r.y & 3, (uint32_t)r.x, id, r.y >> 2 & 2047);
        }
        return h;
    }

    __device__ __forceinline__ int run(rr_instance *I, JobWS &ws, int32_t *log, unsigned logWords, int lineCap,
                                       int32_t *buf, int32_t *ids);
};

template <int MODE>
__device__ __forceinline__ int Sim<MODE>::run(rr_instance *I, JobWS &ws, int32_t *log, unsigned logWords, int lineCap,
                                              int32_t *buf, int32_t *ids)
{
    const int lane = lane_id();
    const unsigned lt = (1u << lane) - 1u;
    const int k = (int)I->n_moves;
    int err = RR_OK;

    // moves without predecessors become statics
    {
        const int n0 = ws.ready0[k];
        for (int b = 0; b < n0; b += 32) {
            const bool c = b + lane < n0;
            const int id = c ? ws.ready0[b + lane] : 0;
            const int4 r = ldg_if(c, rec + 2 * (size_t)id);
            enter(c, r.y & 3, (uint32_t)r.x, id, r.y >> 2 & 2047);
        }
        __syncwarp();
    }
    // the leader: id, direction, position word, clock at the end of its leg,
    // destination row, successors
    int L = -1, d = 0, lend = 0, ldst = 0, nsu = 0, ov = 0;
    uint32_t lpos = 0;
    bool chain = false;       // its only successor is the next id, which waits for nothing else
    int4 s4 = make_int4(0, 0, 0, 0);
    // members: nm of them, of direction dm, on the line `along - clock ==
    // line` (prim) or `across == line`; the clock at their first leg end
    int nm = 0, dm = -1, line = 0, minEnd = INTMAX;
    bool prim = true, changed = false;
    int clk = 0;              // elementary steps so far: also the number of batches
    unsigned nmem = 0;
    // the log: headers from its start, ids from its end
    uint4 *hdr = (uint4 *)log;
    unsigned nseg = 0, idTop = logWords, list = 0;
    // housekeeping every 32 segments (or as many as the log has room for):
    // publish, check the bounds
    int left = min(32, log_room(0u, idTop, lineCap));
    bool logging = left > 0;
    if (!logging) left = 32;
    if (!logging) end_of_log(C);
    long long guard = (g_guard_cap > 0 ? g_guard_cap : I->n_steps + 2ll * k + 16) + 1;
    if (guard < left) left = (int)guard;
    guard -= left;
    // a run is tried with a leader whose predecessor met nothing on its way
    // (elsewhere it would mostly be in vain)
    bool alone = false, tryRun = false;
    // this lane's eight entries of a table's first 256 (a lane beyond the
    // table reads the last eight too: that changes no minimum)
    const int groups = cap >> 3, off = 8 * min(lane, groups - 1);
    const unsigned holders = groups >= 32 ? FULL : (1u << groups) - 1u;      // (lanes of a SIM_SMALL table)

    auto set_leg = [&](uint32_t y) {
        d = (int)(y & 3u);
        lend = clk + (int)(y >> 2 & 2047u);
        ldst = (int)(y >> 13 & 1023u);
        chain = (y >> 23 & 1u) != 0u;
    };
    auto on_clock = [&](uint32_t p) { return (p & 0xffff0000u) | ((p + (uint32_t)clk) & 0xffffu); };
    auto dissolve = [&]() {
        for (int u0 = 0; u0 < nm; u0 += 32) {
            const int u = min(u0 + lane, nm - 1);
            const int2 ie = mie[u];
            enter(u0 + lane < nm, dm, on_clock(mpos[u]), ie.x, ie.y - clk);
        }
        nm = 0;
        minEnd = INTMAX;
        changed = true;
        __syncwarp();
    };
    // the records that come into a run's view, n of them, into L1
    auto look_ahead = [&](int n) {
        touch_rec_if(lane < n, rec, min(L + 2 * RUN - n + lane, k), dump);
    };
    auto housekeeping = [&]() {
        if (guard <= 0) return (int)RR_ERR_TIMEOUT;
        if (*(volatile int *)&C->full) return (int)RR_SIM_RETRY;
        // (a run may have gone beyond the 32)
        guard += left;
        left = 32;
        if (logging) {
            // a header follows the published segments (it says where they
            // end); without room for another one the rest is written here
            if (lane == 0) hdr[nseg] = make_uint4((unsigned)clk, nmem, 0u, 0u);
            __syncwarp();
            __threadfence_block();
            if (lane == 0) *(volatile int *)&C->pub = (int)nseg;
            const int room = log_room(nseg, idTop, lineCap);
            logging = room > 0;
            if (logging) left = min(32, room);
            else end_of_log(C);
        }
        if (guard < left) left = (int)guard;
        guard -= left;
        return (int)RR_OK;
    };
    // the lowest unfinished move, wherever it waits, becomes the leader (rare:
    // nearly always it is released when its predecessor finishes); false when
    // there is none
    auto find_leader = [&]() {
        int best = INTMAX, where = -1, place = 0;
        for (int u = lane; u < nm; u += 32) {
            const int id = mie[u].x;
            if (id < best) { best = id; where = 4; place = u; }
        }
        for (int q = 0; q < 4; ++q)
            for (int e0 = q * cap + 4 * lane; e0 < (q + 1) * cap; e0 += 128) {
                const uint4 a = *(const uint4 *)(pos + e0);
                const uint32_t x[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (x[i] != HOLE && ir[e0 + i].x < best) { best = ir[e0 + i].x; where = q; place = e0 + i; }
            }
        const int least = __reduce_min_sync(FULL, best);
        if (least == INTMAX) return false;
        // (ids are distinct: one lane has it)
        where = (int)uni(best == least ? (uint32_t)where : 0u);
        place = (int)uni(best == least ? (uint32_t)place : 0u);
        L = least;
        const int4 r = rec[2 * (size_t)L];
        s4 = rec[2 * (size_t)L + 1];
        nsu = r.z;
        ov = r.w;
        set_leg(uni((uint32_t)r.y));
        if (where < 4) {
            d = where;
            lpos = uni(pos[place]);
            lend = clk + (int)uni((uint32_t)ir[place].y);
            const int fr = C->nfree[d], tb = d * cap;
            __syncwarp();
            if (lane == 0) {
                pos[place] = HOLE;
                stk[tb + fr] = (uint16_t)(place - tb);
                C->nfree[d] = fr + 1;
            }
        } else {
            d = dm;
            const int2 ie = mie[place];
            lpos = uni(on_clock(mpos[place]));
            lend = (int)uni((uint32_t)ie.y);
            --nm;
            const int2 le = mie[nm];
            const uint32_t lp = mpos[nm];
            __syncwarp();
            if (lane == 0) { mie[place] = le; mpos[place] = lp; }
            __syncwarp();
            int me = INTMAX;
            for (int u = lane; u < nm; u += 32) me = min(me, mie[u].y);
            minEnd = __reduce_min_sync(FULL, me);
            changed = true;
        }
        __syncwarp();
        look_ahead(RUN);
        alone = false;
        return true;
    };

    if (!find_leader() || L != 0) err = RR_ERR_INTERNAL;
    int evEnd = lend;         // the first leg end of the batch
    while (!err) {
        // the statics of the leader's direction: the distance to the nearest
        // line ahead that holds one, 0 when one stands on a line of the leader's
        const int tb = d * cap;
        const uint32_t nadd = 0x10000u - lpos;
        uint4 a = *(const uint4 *)(pos + tb + off), b = *(const uint4 *)(pos + tb + off + 4);
        uint32_t v = min8(a, b, nadd, HOLE);
        if (MODE != SIM_SMALL)
            for (int g = lane + 32; g < groups; g += 32) {
                const uint4 a2 = *(const uint4 *)(pos + tb + 8 * g), b2 = *(const uint4 *)(pos + tb + 8 * g + 4);
                v = min8(a2, b2, nadd, v);
            }
        int fr = C->nfree[d];
        int pick = (int)__reduce_min_sync(FULL, v < 0x10000u ? 0u : v & 0xffffu);
        if (tryRun) {
            tryRun = false;
            int run = 0;
            if (nm == 0 && pick >= lend - clk && guard > 128)
                run = run_of_leaders<MODE>(I, &ws, smem, side, counters, L, d, lend - clk, lpos, clk, nmem, nseg, list, logging);
            if (run > 0) {
                const int segs = run >> 6 & 127, steps = run >> 13;
                L += run & 63;
                if (logging) nseg += (unsigned)segs;
                left -= segs;
                clk += steps;
                nmem += (unsigned)steps;
                const int4 r = rec[2 * (size_t)L];
                lpos = (uint32_t)r.x;
                set_leg((uint32_t)r.y);
                nsu = r.z;
                ov = r.w;
                s4 = rec[2 * (size_t)L + 1];
                look_ahead(run & 63);
                tryRun = (run & 63) == RUN;
                evEnd = lend;
                if (left <= 0) {
                    err = housekeeping();
                    if (err) break;
                }
                continue;
            }
        }
        if (pick == 0) {
            const unsigned ba = __ballot_sync(FULL, (v & 0xffffu) == 0u), bc = __ballot_sync(FULL, v < 0x10000u);
            bool choose;
            if (bc == 0u && (nm == 0 || prim)) choose = true;
            else if (ba == 0u && (nm == 0 || !prim)) choose = false;
            else {
                // candidates on both lines: the smaller smallest id decides
                int ma = INTMAX, mc = INTMAX;
                for (int g = lane; g < groups; g += 32) {
                    const int e = tb + 8 * g;
                    if (MODE != SIM_SMALL) { a = *(const uint4 *)(pos + e); b = *(const uint4 *)(pos + e + 4); }
                    for (unsigned q = match8(a, b, lpos, 0xffffu); q; q &= q - 1) ma = min(ma, ir[e + __ffs(q) - 1].x);
                    for (unsigned q = match8(a, b, lpos, 0xffff0000u); q; q &= q - 1) mc = min(mc, ir[e + __ffs(q) - 1].x);
                }
                for (int u = lane; u < nm; u += 32) {
                    const int id = mie[u].x;
                    if (prim) ma = min(ma, id); else mc = min(mc, id);
                }
                choose = __reduce_min_sync(FULL, ma) < __reduce_min_sync(FULL, mc);
                if (nm > 0 && choose != prim) { dissolve(); fr = C->nfree[d]; }
            }
            alone = false;
            if (choose ? ba : bc) {
                // the chosen line's statics join the members
                int me = minEnd;
                __syncwarp();
                const uint32_t half = choose ? 0xffffu : 0xffff0000u;
                for (int g0 = 0; g0 < groups; g0 += 32) {
                    const int e0 = tb + 8 * (g0 + lane);
                    unsigned q = 0;
                    if (MODE == SIM_SMALL) {
                        q = lane < groups ? match8(a, b, lpos, half) : 0u;
                    } else if (g0 + lane < groups) {
                        q = match8(*(const uint4 *)(pos + e0), *(const uint4 *)(pos + e0 + 4), lpos, half);
                    }
                    for (unsigned bal = MODE == SIM_SMALL ? (choose ? ba : bc) & holders : __ballot_sync(FULL, q != 0u); bal;
                         bal = __ballot_sync(FULL, q != 0u)) {
                        const int n = __popc(bal);
                        if (nm + n > lineCap) { err = RR_ERR_INTERNAL; break; }
                        const bool c = q != 0u;
                        const int i = c ? 31 - __clz(q) : 0, e = e0 + i, rank = __popc(bal & lt), u = nm + rank;
                        q &= ~(1u << i);
                        const int ec = c ? e : tb;
                        const int2 x = ir[ec];
                        const uint32_t p = pos[ec];
                        const int end = x.y + clk;
                        st_if(c, mie + u, x.x, end);
                        st_if(c, mpos + u, (p & 0xffff0000u) | ((p - (uint32_t)clk) & 0xffffu));
                        st_if(c, pos + e, HOLE);
                        st_if(c, stk + tb + fr + rank, e - tb);
                        if (c) me = min(me, end);
                        // its record and its likeliest successor's: read when it finishes
                        touch_rec_if(c, rec, x.x, dump);
                        touch_rec_if(c, rec, x.x + 1, dump);
                        nm += n;
                        fr += n;
                    }
                    if (MODE == SIM_SMALL || err) break;
                }
                if (err) break;
                if (lane == 0) C->nfree[d] = fr;
                minEnd = __reduce_min_sync(FULL, me);
                prim = choose;
                dm = d;
                line = choose ? (int)(lpos & 0xffffu) - clk : (int)(lpos >> 16);
                changed = true;
                __syncwarp();
            }
            evEnd = min(lend, minEnd);
            // the nearest line ahead of the leader's own (those that have just
            // joined along its line of motion are further than its leg's end)
            v = min8(a, b, nadd - 1u, HOLE);
            if (MODE != SIM_SMALL)
                for (int g = lane; g < groups; g += 32) {
                    const uint4 a2 = *(const uint4 *)(pos + tb + 8 * g), b2 = *(const uint4 *)(pos + tb + 8 * g + 4);
                    v = min8(a2, b2, nadd - 1u, v);
                }
            pick = (int)__reduce_min_sync(FULL, v & 0xffffu) + 1;
        }
        // the segment: up to the first leg end or the nearest line ahead
        const int kseg = min(pick, evEnd - clk);
        if (logging) {
            if (changed) {
                changed = false;
                idTop -= (unsigned)nm;
                list = idTop;
                // (lanes beyond the members read room that nothing uses)
                const int id = mie[lane].x;
                if (lane < nm) log[list + lane] = id;
                if (nm > 32)
                    for (int u = 32 + lane; u < nm; u += 32) log[list + u] = mie[u].x;
            }
            if (lane == 0) hdr[nseg] = make_uint4((unsigned)clk, nmem, list, (unsigned)L | (unsigned)d << 30);
            ++nseg;
        } else {
            const unsigned long long o1 = (unsigned long long)clk + kseg, m1 = nmem + (unsigned long long)kseg * (nm + 1);
            if (o1 <= room_of(I->cap_ops) && m1 <= room_of(I->cap_members)) {
                for (int u = lane; u < nm; u += 32) ids[u] = mie[u].x;
                __syncwarp();
                if constexpr (MODE == SIM_SMALL)
                    write_segment(as_global(I->ops), as_global(I->members), OpLane(lane), (unsigned)clk, nmem, kseg, nm + 1, d, L,
                                  ids, buf);
                else write_call(I, (unsigned)clk, nmem, kseg, nm + 1, d, L, ids, buf);
            }
        }
        // everything in the batch advances
        nmem += (unsigned)(kseg * (nm + 1));
        clk += kseg;
        lpos += (uint32_t)kseg;
        if (--left <= 0) {
            err = kseg < 1 ? RR_ERR_INTERNAL : housekeeping();
            if (err) break;
        }
        if (clk != evEnd) { alone = false; continue; }
        bool fin = false, moved = false;
        int4 nr = make_int4(0, 0, 0, 0), ns4 = nr;
        if (clk == lend) {
            // the next id's record (an entry beyond the last one exists)
            nr = rec[2 * (size_t)(L + 1)];
            ns4 = rec[2 * (size_t)(L + 1) + 1];
            moved = true;
            if (d < 2 || ldst == (int)(lpos >> 16) - 1) fin = true;
            else {
                const Leg g = second_leg(d, lpos, ldst);
                d = g.d; lpos = g.pos; lend = clk + g.rem;
            }
        }
        // once the leader has finished, the next id (if it becomes ready now)
        // is the next leader and enters no table
        const int handId = fin ? L + 1 : -1;
        bool hand = false;
        if (clk == minEnd) {
            // members whose leg ended leave: they turn (into the tables) or
            // finish (and release their successors)
            int nk = 0, me = INTMAX;
            for (int u0 = 0; u0 < nm; u0 += 32) {
                const int u = u0 + lane;
                const bool act = u < nm;
                const int2 ie = mie[act ? u : u0];
                const uint32_t p = mpos[act ? u : u0];
                const bool ended = act && ie.y == clk, keep = act && ie.y != clk;
                int4 r = ldg_if(ended, rec + 2 * (size_t)ie.x), s = ldg_if(ended, rec + 2 * (size_t)ie.x + 1);
                const unsigned kb = __ballot_sync(FULL, keep);
                me = keep ? min(me, ie.y) : me;
                const int w = nk + __popc(kb & lt);
                if (nk != u0 || kb != FULL) {                          // some move up
                    __syncwarp();
                    st_if(keep, mie + w, ie.x, ie.y);
                    st_if(keep, mpos + w, p);
                    if (nm <= 32 || __any_sync(FULL, ended)) {
                        if (dm >= 2) {
                            const int dst = r.y >> 13 & 1023;
                            const bool turn = ended && dst != (int)(p >> 16) - 1;
                            const Leg g = second_leg(dm, on_clock(p), dst);
                            enter(turn, g.d, g.pos, ie.x, g.rem);
                            if (turn) r.z = 0;
                        }
                        const int most = (int)uni((uint32_t)r.z);
                        for (int e = 0; e < most; ++e) {
                            int32_t v = e == 0 ? s.x : e == 1 ? s.y : e == 2 ? s.z : s.w;
                            if (e >= 4) v = ldg_if(e < r.z, (const void *)(succ + r.w + e - 4));
                            hand |= release(e < r.z, v, handId);
                        }
                    }
                    __syncwarp();
                }
                nk += __popc(kb);
            }
            nm = nk;
            minEnd = __reduce_min_sync(FULL, me);
            changed = true;
        }
        if (fin) {
            if (chain) hand = true;
            else {
                const int n = (int)uni((uint32_t)nsu);
                for (int e0 = 0; e0 < n; e0 += 32) {
                    const int e = e0 + lane;
                    int32_t v = e == 0 ? s4.x : e == 1 ? s4.y : e == 2 ? s4.z : s4.w;
                    if (n > 4) {
                        const int w = ldg_if(e >= 4 && e < n, (const void *)(succ + ov + e - 4));
                        v = e >= 4 ? w : v;
                    }
                    hand |= release(e < n, v, handId);
                }
                hand = __any_sync(FULL, hand);
                __syncwarp();
            }
            if (hand) {
                L = handId;
                lpos = (uint32_t)nr.x;
                set_leg((uint32_t)nr.y);
                nsu = nr.z;
                ov = nr.w;
                s4 = ns4;
                look_ahead(1);
                tryRun = alone;
                alone = true;
            } else if (!find_leader()) {
                break;
            }
        }
        // members no longer on the leader's line or in its direction?
        if (moved && nm > 0 && !(dm == d && line == (prim ? (int)(lpos & 0xffffu) - clk : (int)(lpos >> 16)))) dissolve();
        evEnd = min(lend, minEnd);
    }
    return sim_end(I, C, hdr, nseg, logging, clk, nmem, err);
}

// ------------------------------------------------- the wide simulation
//
// For instances with more ready moves of a direction than the tables hold (no
// planner here makes such lists; rr_batch takes any path system): statics by
// the vertex that they stand on (ready moves share none), with room for every
// move, so that a segment's cost grows with the grid's side and not with the
// length of the list. A line's statics are found by reading the line; counts
// of every line say whether there are any, a bit per line of a direction where
// the next one ahead is. Against a table of all legs in global memory, scanned
// whole at every segment: 524 288 dominoes on 1024 x 1024 (1 278 batches) 3.2 s
// -> 60 ms, 600 000 moves of one token beside 512 others 31 s -> 0.9 s.

constexpr uint32_t NOBODY = 0xffffffffu;
struct Wide {
    uint32_t *map;            // m * n: id and direction (upper two bits) of the static on a vertex
                              // (where the first horizontal coverers were: the conflict graph is done)
    int2 *state;              // k: a static's position word, steps left and direction (two bits);
                              // .y is 0 for a move that waits or is a member, -1 for a finished one
    int32_t *al, *ac;         // 4 * side each: statics of a direction on a line across its way, along it
    uint32_t *some;           // 4 * 32: which lines across a direction's way hold any
    int m, n, side;

    // (where the tables were: 14 words for each of at least max(side, 56) entries)
    static __device__ size_t shared_words(int side) { return 8 * (size_t)side + 128; }
    __device__ __forceinline__ Wide(rr_instance *I, const JobWS &ws, char *smem, int side_)
        : map((uint32_t *)as_global(ws.firstH)), state(as_global(ws.state)), m(I->m), n(I->n), side(side_)
    {
        al = (int32_t *)smem;
        ac = al + 4 * side;
        some = (uint32_t *)(ac + 4 * side);
    }
    // A position's line across the way (numbered along it) and along it, its
    // row and column.
    __device__ __forceinline__ int line_al(int d, uint32_t p) const
    {
        return (int)(p & 0xffffu) - ((d & 1) ? 1 : MIRROR - side);
    }
    __device__ __forceinline__ int line_ac(uint32_t p) const { return (int)(p >> 16) - 1; }
    __device__ __forceinline__ int coord(int d, uint32_t p) const
    {
        return (d & 1) ? (int)(p & 0xffffu) - 1 : MIRROR - 1 - (int)(p & 0xffffu);
    }
    __device__ __forceinline__ int row(int d, uint32_t p) const { return d < 2 ? coord(d, p) : line_ac(p); }
    __device__ __forceinline__ int col(int d, uint32_t p) const { return d < 2 ? line_ac(p) : coord(d, p); }

    // A move becomes a static, or is one no longer (each lane its own).
    __device__ __forceinline__ void put(int d, uint32_t p, int id, int rem)
    {
        const int a = line_al(d, p);
        map[(size_t)row(d, p) * n + col(d, p)] = (uint32_t)id | (uint32_t)d << 30;
        state[id] = make_int2((int)p, rem << 2 | d);
        if (atomicAdd(&al[d * side + a], 1) == 0) atomicOr(&some[32 * d + (a >> 5)], 1u << (a & 31));
        atomicAdd(&ac[d * side + line_ac(p)], 1);
    }
    __device__ __forceinline__ void take(int d, uint32_t p, int id)
    {
        const int a = line_al(d, p);
        map[(size_t)row(d, p) * n + col(d, p)] = NOBODY;
        state[id].y = 0;
        if (atomicSub(&al[d * side + a], 1) == 1) atomicAnd(&some[32 * d + (a >> 5)], ~(1u << (a & 31)));
        atomicSub(&ac[d * side + line_ac(p)], 1);
    }
    // Lines from p's to the next one ahead that holds a static of direction d
    // (far, if there is none).
    __device__ __forceinline__ int ahead(int d, uint32_t p) const
    {
        const int lane = lane_id(), a = line_al(d, p), w = a >> 5;
        uint32_t x = some[32 * d + lane];
        x &= lane < w ? 0u : lane == w ? ~(((2u << (a & 31)) - 1u)) : FULL;
        const unsigned b = __ballot_sync(FULL, x != 0u);
        if (!b) return 0x7fff;
        const int src = __ffs(b) - 1;
        return 32 * src + __ffs(__shfl_sync(FULL, x, src)) - 1 - a;
    }
    // f(lane's static there or not, its id) for the vertices of p's line
    // across the way of d (or along it), 32 at a time, four loads in flight.
    template <class F>
    __device__ __forceinline__ void line(int d, uint32_t p, bool across, F f) const
    {
        const bool isRow = across == (d < 2);
        const int len = isRow ? n : m, step = isRow ? 1 : n;
        const uint32_t *at = map + (isRow ? (size_t)row(d, p) * n : (size_t)col(d, p));
        for (int i0 = lane_id(); i0 - lane_id() < len; i0 += 128) {
            uint32_t w[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) w[u] = i0 + 32 * u < len ? at[(size_t)(i0 + 32 * u) * step] : NOBODY;
#pragma unroll
            for (int u = 0; u < 4; ++u) f(w[u] != NOBODY && (int)(w[u] >> 30) == d, (int)(w[u] & 0x3fffffffu));
        }
    }
    __device__ __forceinline__ int least_id(int d, uint32_t p, bool across) const
    {
        int least = INTMAX;
        line(d, p, across, [&](bool c, int id) { least = c ? min(least, id) : least; });
        return least;
    }
};

// The simulation over such a map: as Sim, without what makes that one fast on
// plans (runs of leaders, counters in shared memory).
struct WideSim : Wide {
    int2 *mie;                // members: id, clock at the end of the leg
    uint32_t *mpos;           // members: position word, `along` minus the clock
    SimCtl *C;
    const int4 *rec;
    const int32_t *succ;
    const int2 *multiMove;
    int32_t *multi;
    uint32_t dump;

    using Wide::Wide;

    __device__ __forceinline__ bool release(bool c, int32_t v, int handId)
    {
        const bool single = c && (v & SUCC_SINGLE);
        int id = v & SUCC_ID, y = 0;
        uint32_t p = 0;
        bool ready = single;
        if (single) {
            const int4 r = rec[2 * (size_t)id];
            p = (uint32_t)r.x;
            y = r.y;
        } else if (c && (atomicSub(&multi[id], 1) & MULTI_COUNT) == 1) {
            y = ldg_volatile_if(true, multi + id) >> MULTI_BITS;
            const int2 mv = multiMove[id];
            id = mv.x;
            p = (uint32_t)mv.y;
            ready = true;
        }
        __syncwarp();
        const bool h = ready && id == handId;
        if (ready && !h) put(y & 3, p, id, y >> 2 & 2047);
        __syncwarp();
        return h;
    }

    __device__ __forceinline__ int run(rr_instance *I, JobWS &ws, int32_t *log, unsigned logWords, int lineCap,
                                       int32_t *buf, int32_t *ids);
};

__device__ __forceinline__ int WideSim::run(rr_instance *I, JobWS &ws, int32_t *log, unsigned logWords, int lineCap,
                                            int32_t *buf, int32_t *ids)
{
    const int lane = lane_id();
    const unsigned lt = (1u << lane) - 1u;
    const int k = (int)I->n_moves;
    int err = RR_OK;

    // moves without predecessors become statics
    for (int b = lane, n0 = ws.ready0[k]; b < n0; b += 32) {
        const int id = ws.ready0[b];
        const int4 r = rec[2 * (size_t)id];
        put(r.y & 3, (uint32_t)r.x, id, r.y >> 2 & 2047);
    }
    __syncwarp();
    // leader, members, clock and log as in Sim
    int L = -1, d = 0, lend = 0, ldst = 0, nsu = 0, ov = 0;
    uint32_t lpos = 0;
    int4 s4 = make_int4(0, 0, 0, 0);
    int nm = 0, dm = -1, line_ = 0, minEnd = INTMAX;
    bool prim = true, changed = false;
    int clk = 0;
    unsigned nmem = 0;
    uint4 *hdr = (uint4 *)log;
    unsigned nseg = 0, idTop = logWords, list = 0;
    int left = min(32, log_room(0u, idTop, lineCap));
    bool logging = left > 0;
    if (!logging) { left = 32; end_of_log(C); }
    long long guard = (g_guard_cap > 0 ? g_guard_cap : I->n_steps + 2ll * k + 16) + 1;
    if (guard < left) left = (int)guard;
    guard -= left;

    auto set_record = [&](const int4 r, const int4 s) {
        d = (int)uni((uint32_t)r.y & 3u);
        lpos = uni((uint32_t)r.x);
        lend = clk + (r.y >> 2 & 2047);
        ldst = r.y >> 13 & 1023;
        nsu = r.z;
        ov = r.w;
        s4 = s;
    };
    auto on_clock = [&](uint32_t p) { return (p & 0xffff0000u) | ((p + (uint32_t)clk) & 0xffffu); };
    auto dissolve = [&]() {
        for (int u = lane; u < nm; u += 32) put(dm, on_clock(mpos[u]), mie[u].x, mie[u].y - clk);
        nm = 0;
        minEnd = INTMAX;
        changed = true;
        __syncwarp();
    };
    // the lowest unfinished move becomes the leader: every id up to the last
    // leader's has finished, so on from there
    auto find_leader = [&]() {
        unsigned open = 0;
        int b = L + 1;
        for (; b < k; b += 32) {
            open = __ballot_sync(FULL, b + lane < k && state[min(b + lane, k - 1)].y >= 0);
            if (open) break;
        }
        if (!open) return false;
        L = b + __ffs(open) - 1;
        set_record(rec[2 * (size_t)L], rec[2 * (size_t)L + 1]);
        const int2 st = state[L];
        __syncwarp();
        if (st.y > 0) {
            d = (int)uni((uint32_t)st.y & 3u);
            lpos = uni((uint32_t)st.x);
            lend = clk + (st.y >> 2);
            if (lane == 0) take(d, lpos, L);
        } else {
            int at = -1;
            for (int u = lane; u < nm; u += 32) at = mie[u].x == L ? u : at;
            at = __reduce_max_sync(FULL, at);
            if (at < 0) return false;               // neither ready nor moving
            d = dm;
            lpos = uni(on_clock(mpos[at]));
            lend = mie[at].y;
            --nm;
            const int2 le = mie[nm];
            const uint32_t lp = mpos[nm];
            __syncwarp();
            if (lane == 0) { mie[at] = le; mpos[at] = lp; }
            __syncwarp();
            int me = INTMAX;
            for (int u = lane; u < nm; u += 32) me = min(me, mie[u].y);
            minEnd = __reduce_min_sync(FULL, me);
            changed = true;
        }
        __syncwarp();
        return true;
    };

    if (!find_leader() || L != 0) err = RR_ERR_INTERNAL;
    while (!err) {
        const int la = d * side + line_al(d, lpos), lc = d * side + line_ac(lpos);
        const bool onA = al[la] != 0, onC = ac[lc] != 0;
        if (onA || onC) {
            bool choose;
            if (!onC && (nm == 0 || prim)) choose = true;
            else if (!onA && (nm == 0 || !prim)) choose = false;
            else {
                // candidates on both lines: the smaller smallest id decides
                int ma = least_id(d, lpos, true), mc = least_id(d, lpos, false);
                for (int u = lane; u < nm; u += 32) {
                    const int id = mie[u].x;
                    if (prim) ma = min(ma, id); else mc = min(mc, id);
                }
                choose = __reduce_min_sync(FULL, ma) < __reduce_min_sync(FULL, mc);
                if (nm > 0 && choose != prim) dissolve();
            }
            if (choose ? onA : onC) {
                // the chosen line's statics join the members
                int me = minEnd;
                __syncwarp();
                line(d, lpos, choose, [&](bool c, int id) {
                    const unsigned bal = __ballot_sync(FULL, c);
                    const int u = nm + __popc(bal & lt);
                    if (nm + __popc(bal) > lineCap) { err = RR_ERR_INTERNAL; return; }
                    if (c) {
                        const int2 st = state[id];
                        const uint32_t p = (uint32_t)st.x;
                        const int end = (st.y >> 2) + clk;
                        mie[u] = make_int2(id, end);
                        mpos[u] = (p & 0xffff0000u) | ((p - (uint32_t)clk) & 0xffffu);
                        take(d, p, id);
                        me = min(me, end);
                    }
                    nm += __popc(bal);
                });
                if (err) break;
                minEnd = __reduce_min_sync(FULL, me);
                prim = choose;
                dm = d;
                line_ = choose ? (int)(lpos & 0xffffu) - clk : (int)(lpos >> 16);
                changed = true;
                __syncwarp();
            }
        }
        // the segment: up to the first leg end or the nearest line ahead
        const int evEnd = min(lend, minEnd), kseg = min(ahead(d, lpos), evEnd - clk);
        if (kseg < 1) { err = RR_ERR_INTERNAL; break; }
        if (logging) {
            if (changed) {
                changed = false;
                idTop -= (unsigned)nm;
                list = idTop;
                for (int u = lane; u < nm; u += 32) log[list + u] = mie[u].x;
            }
            if (lane == 0) hdr[nseg] = make_uint4((unsigned)clk, nmem, list, (unsigned)L | (unsigned)d << 30);
            ++nseg;
        } else {
            const unsigned long long o1 = (unsigned long long)clk + kseg, m1 = nmem + (unsigned long long)kseg * (nm + 1);
            if (o1 <= room_of(I->cap_ops) && m1 <= room_of(I->cap_members)) {
                for (int u = lane; u < nm; u += 32) ids[u] = mie[u].x;
                __syncwarp();
                write_call(I, (unsigned)clk, nmem, kseg, nm + 1, d, L, ids, buf);
            }
        }
        // everything in the batch advances
        nmem += (unsigned)(kseg * (nm + 1));
        clk += kseg;
        lpos += (uint32_t)kseg;
        if (--left <= 0) {
            if (guard <= 0) { err = RR_ERR_TIMEOUT; break; }
            left = 32;
            if (logging) {
                if (lane == 0) hdr[nseg] = make_uint4((unsigned)clk, nmem, 0u, 0u);
                __syncwarp();
                __threadfence_block();
                if (lane == 0) *(volatile int *)&C->pub = (int)nseg;
                const int room = log_room(nseg, idTop, lineCap);
                logging = room > 0;
                if (logging) left = min(32, room);
                else end_of_log(C);
            }
            if (guard < left) left = (int)guard;
            guard -= left;
        }
        if (clk != evEnd) continue;
        bool fin = false, moved = false;
        if (clk == lend) {
            moved = true;
            if (d < 2 || ldst == (int)(lpos >> 16) - 1) fin = true;
            else {
                const Leg g = second_leg(d, lpos, ldst);
                d = g.d; lpos = g.pos; lend = clk + g.rem;
            }
        }
        const int handId = fin ? L + 1 : -1;       // the next leader, if it becomes ready now
        bool hand = false;
        if (clk == minEnd) {
            // members whose leg ended leave: they turn or finish
            int nk = 0, me = INTMAX;
            for (int u0 = 0; u0 < nm; u0 += 32) {
                const int u = u0 + lane;
                const int2 ie = mie[min(u, nm - 1)];
                const uint32_t p = mpos[min(u, nm - 1)];
                const bool ended = u < nm && ie.y == clk, keep = u < nm && ie.y != clk;
                const unsigned kb = __ballot_sync(FULL, keep);
                const int w = nk + __popc(kb & lt);
                if (keep) { mie[w] = ie; mpos[w] = p; me = min(me, ie.y); }
                int4 r = make_int4(0, 0, 0, 0), s = r;
                if (ended) {
                    r = rec[2 * (size_t)ie.x];
                    s = rec[2 * (size_t)ie.x + 1];
                    const int dst = r.y >> 13 & 1023;
                    if (dm >= 2 && dst != (int)(p >> 16) - 1) {
                        const Leg g = second_leg(dm, on_clock(p), dst);
                        put(g.d, g.pos, ie.x, g.rem);
                        r.z = 0;
                    } else {
                        state[ie.x].y = -1;
                    }
                }
                __syncwarp();
                const int most = (int)uni((uint32_t)r.z);
                for (int e = 0; e < most; ++e) {
                    int32_t v = e == 0 ? s.x : e == 1 ? s.y : e == 2 ? s.z : s.w;
                    if (e >= 4 && e < r.z) v = succ[r.w + e - 4];
                    hand |= release(e < r.z, v, handId);
                }
                nk += __popc(kb);
            }
            nm = nk;
            minEnd = __reduce_min_sync(FULL, me);
            changed = true;
        }
        if (fin) {
            const int n_ = (int)uni((uint32_t)nsu);
            for (int e0 = 0; e0 < n_; e0 += 32) {
                const int e = e0 + lane;
                int32_t v = e == 0 ? s4.x : e == 1 ? s4.y : e == 2 ? s4.z : s4.w;
                if (e >= 4 && e < n_) v = succ[ov + e - 4];
                hand |= release(e < n_, v, handId);
            }
            if (__any_sync(FULL, hand)) {
                L = handId;
                set_record(rec[2 * (size_t)L], rec[2 * (size_t)L + 1]);
                touch_rec_if(lane == 0, rec, min(L + 1, k), dump);
            } else if (!find_leader()) {
                break;
            }
        }
        // members no longer on the leader's line or in its direction?
        if (moved && nm > 0 && !(dm == d && line_ == (prim ? (int)(lpos & 0xffffu) - clk : (int)(lpos >> 16)))) dissolve();
    }
    return sim_end(I, C, hdr, nseg, logging, clk, nmem, err);
}

// The fields that both forms have, and the log: the chains of the conflict
// graph are no longer needed.
template <class SIM>
__device__ __forceinline__ int sim_run(SIM &S, rr_instance *I, JobWS &ws, const SimLayout &Y)
{
    S.mie = Y.mie; S.mpos = Y.mpos; S.C = Y.C;
    S.rec = as_global(ws.rec); S.succ = as_global(ws.succ); S.multi = as_global(ws.multi);
    S.multiMove = as_global(ws.multiMove);
    S.dump = sh_addr(Y.dump);
    return S.run(I, ws, as_global(ws.nextAt), (unsigned)((4 * (ws.P + 1) + 255) / 256 * 64), Y.MC, Y.bufs, Y.ids);
}

// A simulation starts: its control words (every thread calls it).
__device__ __forceinline__ void ctl_begin(SimCtl *C, int free)
{
    if (threadIdx.x < 4) C->nfree[threadIdx.x] = free;
    if (threadIdx.x == 0) {
        C->full = C->pub = C->next = C->fin = 0;
        C->status = RR_OK;
    }
}
// The counters in shared memory.
__device__ __forceinline__ void counters_begin(const SimLayout &Y, const JobWS &ws, int counters)
{
    unsigned short *c16 = (unsigned short *)Y.cnt;
    const int ncnt = min(counters, ws.nmulti);
    for (int i = threadIdx.x; i < ncnt; i += blockDim.x) c16[i] = (unsigned short)(ws.multi[i] & MULTI_COUNT);
}

// Warp 0 runs simulate(), the others write, warp 0 writes too once it is done.
// Returns the status (every thread calls it).
template <class F>
__device__ __forceinline__ int sim_and_write(F simulate, rr_instance *I, JobWS &ws, const SimLayout &Y, int side)
{
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (wid == 0) {
        const int st = simulate();
        if (lane == 0) Y.C->status = st;
        __syncwarp();
    }
    run_writers(Y.C, I, as_global(ws.nextAt), Y.bufs + sim_pow2(side) * wid);
    __syncthreads();
    return Y.C->status;
}

// An instance that outgrew the tables starts over in the wide form (the
// batches written so far are the same ones): its state at the start, for the
// whole block, its simulation, both with writers. Out of line: in line, the
// registers and the stack of this form would cost the other one.
static __device__ __noinline__ void wide_begin(rr_instance *I, JobWS *ws, char *smem, int side)
{
    const Wide W(I, *ws, smem, side);
    const int k = (int)I->n_moves;
    for (int i = threadIdx.x; i < W.m * W.n; i += blockDim.x) W.map[i] = NOBODY;
    for (int b = threadIdx.x; b < k; b += blockDim.x) W.state[b] = make_int2(0, 0);
    for (int i = threadIdx.x; i < (int)Wide::shared_words(side); i += blockDim.x) W.al[i] = 0;
    // (the first form counted in-degrees down)
    for (int x = threadIdx.x; x < ws->nmulti; x += blockDim.x)
        ws->multi[x] = (ws->multi[x] & ~MULTI_COUNT) | ws->indeg[ws->multiMove[x].x];
}
static __device__ __noinline__ int wide_run(rr_instance *I, JobWS *ws, char *smem, int side)
{
    WideSim S(I, *ws, smem, side);
    return sim_run(S, I, *ws, SimLayout(smem, side));
}
static __device__ __noinline__ int wide_block(rr_instance *I, JobWS *ws, char *smem, int side)
{
    const SimLayout Y(smem, side);
    __syncthreads();                    // every thread has read the first form's status
    ctl_begin(Y.C, 0);
    wide_begin(I, ws, smem, side);
    return sim_and_write([&]() { return wide_run(I, ws, smem, side); }, I, *ws, Y, side);
}

// The simulation of one instance by one block (every thread calls it). A block
// without writers is one warp; s_wide follows for the instances that outgrew the
// tables, s_write writes afterwards.
template <int MODE, bool WRITERS>
__device__ __forceinline__ void sim_block(rr_instance *I, JobWS &ws, char *smem, int side, int counters)
{
    const int k = (int)I->n_moves;
    if (!live(I)) return;                       // the same in every thread: set before this kernel or a barrier
    if (k == 0) {
        if (threadIdx.x == 0) { I->n_ops = 0; I->n_members = 0; }
        return;
    }
    const int cap = sim_cap(side);
    const SimLayout Y(smem, side);
    Sim<MODE> S;
    S.pos = (uint32_t *)smem;
    S.ir = (int2 *)(S.pos + 4 * cap);
    S.stk = (uint16_t *)(S.ir + 4 * cap);
    S.cap = cap;
    S.cnt = Y.cnt;
    S.ncnt = min(counters, ws.nmulti);
    S.allShared = counters >= ws.nmulti;
    S.smem = smem; S.side = side; S.counters = counters;
    auto tables_begin = [&]() {                 // entries are handed out from a table's start
        for (int i = threadIdx.x; i < 4 * cap; i += blockDim.x) {
            S.pos[i] = HOLE;
            S.stk[i] = (uint16_t)(cap - 1 - i % cap);
        }
    };
    int st;
    if constexpr (WRITERS) {
        ctl_begin(Y.C, cap);
        tables_begin();
        counters_begin(Y, ws, counters);
        st = sim_and_write([&]() { return sim_run(S, I, ws, Y); }, I, ws, Y, side);
        if (st == RR_SIM_RETRY && k >= SIM_WIDE_MIN) st = wide_block(I, &ws, smem, side);
    } else {
        ctl_begin(Y.C, cap);
        tables_begin();
        counters_begin(Y, ws, counters);
        __syncthreads();
        st = sim_run(S, I, ws, Y);
        if (threadIdx.x == 0) ws.nseg = Y.C->pub;        // s_write follows
        if (st == RR_SIM_RETRY && k >= SIM_WIDE_MIN) {
            if (threadIdx.x == 0) I->status = RR_SIM_RETRY;      // s_wide takes over
            return;
        }
    }
    if (threadIdx.x == 0 && st != RR_OK) I->status = st == RR_SIM_RETRY ? RR_ERR_INTERNAL : st;
}

// The instances that outgrew the tables in blocks of one warp. A kernel of its
// own, whose blocks nearly always return at once: with both forms in one kernel
// the first one's code is slower whatever way the second is called (4096 mixed
// grids 38.2 ms, 35.0 this way; 2 000 of sides 64 to 128 11.1 and 10.2).
__device__ inline void s_wide(rr_instance *I, JobWS &ws, char *smem, int side)
{
    if (I->status != RR_SIM_RETRY) return;
    __syncthreads();
    const SimLayout Y(smem, side);
    if (threadIdx.x == 0) I->status = RR_OK;
    ctl_begin(Y.C, 0);
    wide_begin(I, &ws, smem, side);
    __syncthreads();
    const int st = wide_run(I, &ws, smem, side);
    if (threadIdx.x == 0) {
        ws.nseg = Y.C->pub;
        if (st != RR_OK) I->status = st == RR_SIM_RETRY ? RR_ERR_INTERNAL : st;
    }
}

} // namespace rrk
