// rr_internal.cuh -- device-side types and helpers shared by the kernels of
// the red-rec planner and batching routine (arXiv 2504.06182, Alg. 1 and 2).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>
#include "rr.h"

namespace rrk {

constexpr unsigned FULL = 0xffffffffu;

// Block coordinates of a stage (the stage functions of rr_plan.cuh,
// rr_bird.cuh and rr_batch.cuh): the hardware's when a stage runs as a
// kernel of its own; x = 0, gx = 1 when one block runs the whole path of one
// grid (the single-grid kernel), so that every grid-stride loop covers all
// of its items. Stages that give a warp an item use w and nw: this warp's
// first item and the number of warps on this instance.
struct Blk { int x, y, gx, w, nw; };
__device__ __forceinline__ Blk hw_blk()
{
    const int wpb = blockDim.x >> 5;
    return Blk{(int)blockIdx.x, (int)blockIdx.y, (int)gridDim.x, (int)blockIdx.x * wpb + (int)(threadIdx.x >> 5),
               (int)gridDim.x * wpb};
}
// The same with `per` warps of a block on each instance, hence several
// instances per block: for calls over very many grids, whose instances would
// otherwise take a whole block each, most of it idle when they are narrow.
__device__ __forceinline__ Blk hw_blk_shared(int per)
{
    const int wpb = blockDim.x >> 5, wid = threadIdx.x >> 5;
    return Blk{(int)blockIdx.x, (int)blockIdx.y * (wpb / per) + wid / per, (int)gridDim.x,
               (int)blockIdx.x * per + wid % per, (int)gridDim.x * per};
}

// Column classification after the column phase (Alg. 1 first loop, solved for
// every column of non-negative surplus at once as in Sec. III.D).
enum ColKind : int32_t {
    KIND_TARGET_SOLVED = 0,   // target column, surplus >= 0: exact 1D window solve
    KIND_RECEIVER = 1,        // target column, surplus < 0
    KIND_OUTER_FULL = 2,      // outside the target columns, enough atoms to fill its reservoir cells
    KIND_OUTER_PART = 3       // outside the target columns, fewer atoms than reservoir cells
};

struct ColInfo {
    int32_t K, ntop, nband, nbot;   // atoms: all, rows < r0, rows in [r0, r1), rows >= r1
    int32_t sigma;                  // surplus after the column phase
    int32_t kind;
    int32_t ptop, pbot;             // donatable pool sizes (nearest-to-band first)
    int32_t tbase, bbase;           // atom index of the nearest top / bottom pool atom
    int32_t a;                      // target solved: top atoms taken into the window
    int32_t kd_end, ku_start;       // solve order ranges (see emission)
    int32_t nmoves;                 // moves of this column's column-phase unit
    int32_t topRun, botRun;         // outer full: atoms already on their virtual targets
};

// One pairing iteration (Alg. 1 main loop).
struct Event {
    int32_t kase;       // 1: receiver saturated, 2: both saturated, 3: donor exhausted (delayed)
    int32_t i, j;       // donor, receiver
    int32_t x, a;       // tokens exchanged, of which a come from above the band
    int32_t t0, b0;     // donor pool cursors (nearest-first index) before the exchange
    int32_t at;         // of the p-th slot: the event there when ordered by receiver (saturation
                        // order) and, within a receiver, by time
};

// A receiver unit, in the order receivers become saturated.
struct RecvInfo {
    int32_t j;
    int32_t ev_first;   // its events' first slot (Event::at)
    int32_t ncontrib;   // its events
    int32_t nT;         // sources above the band (mandatory + chosen)
    int32_t kd_end, ku_start, nmoves;
    int32_t pad;
};

// Shared memory of the pairing stage per column.
constexpr int PAIR_BYTES = 42;

struct Arena {
    char *base;
    unsigned long long size;
    unsigned long long *top;   // device bump pointer
};

struct JobWS {
    // planning
    uint32_t *colbits;     // n * W, column-major bit columns (bit r & 31 of word r >> 5)
    int16_t *atomRows;     // n * m: rows of the atoms of each column, ascending
    int16_t *holeRows;     // n * h: rows of the empty band traps of each column, ascending
    ColInfo *col;          // n
    RecvInfo *recv;        // n
    Event *ev;             // n + 1
    int32_t *unitOff;      // 2n + 1
    int32_t nrecv, nev;
    int32_t npending, pending;   // calls over many grids: how many still need pairing (of the first
                                 // instance), the i-th of them
    int32_t nlacking, lacking;   // how many have receiver units (of the first instance), the i-th of them
    // batching (Gamma + simulation)
    int64_t P;             // total path vertices (sum of path length + 1)
    int32_t *pairOff;      // k + 1
    int32_t *nextAt;       // P
    int32_t *succ;         // P: a path's successors at its vertex offset (pairOff)
    int32_t *indeg;        // k
    int4 *rec;             // 2 (k + 1), the last two unused: see move_rec
    int32_t *ready0;       // k + 1: moves without predecessors; [k] = their count
    // Gamma by sweeps: moves ending in each column, L-moves starting on each row
    int32_t *colOff, *colCur, *colList;   // n + 1, n, k
    int32_t *rowOff, *rowCur, *rowList;   // m + 1, m, k
    int32_t *firstH;       // m * n: lowest-id L-move crossing each vertex, -1
    int2 *state;           // k: the wide simulation's moves (Wide)
    // the moves with several predecessors, by number: in-degree and first leg
    // (MULTI_BITS), id, position word
    int32_t *multi;
    int2 *multiMove;
    int32_t *multiNo;      // k: a move's number among them
    int32_t nmulti;        // how many there are
    int32_t nseg;          // logged segments that are still to be written
    // path-vertex offsets by the multi-block scan (large move lists only):
    // one status word per tile, the tile counter
    unsigned long long *lbStatus;
    int32_t *lbCounter;
};

// Multi-block single-pass scan (decoupled look-back) of the path-vertex
// offsets: tiles of LB_TILE moves, taken in order from a per-instance
// counter by blocks of LB_THREADS threads; used for move lists of at least
// LB_MIN_MOVES (below that one block scans them).
constexpr int LB_THREADS = 512, LB_ITEMS = 8, LB_TILE = LB_THREADS * LB_ITEMS;
constexpr int64_t LB_MIN_MOVES = 1 << 16;

// Side bound of simulation size class c of nclass over grids up to
// max_side (the last class takes max_side itself).
__host__ __device__ inline int class_side(int max_side, int c, int nclass)
{
    if (c >= nclass - 1) return max_side;
    const int s = (max_side * (c + 1) + nclass - 1) / nclass;
    return s < 32 ? 32 : s;
}

// Block-wide state of a simulation in shared memory.
struct SimCtl {
    int nfree[4];             // free entries of each direction's table
    int full;                 // a table was full
    int pub;                  // segments of the log that the writers may write
    int next;                 // first segment not yet taken by a writer (by 32)
    int fin;                  // pub is final: the simulation, or its log, has ended
    int status;               // its end: RR_OK, RR_SIM_RETRY or an error
    int pad[3];
};

// Table entries per direction in shared memory. Red-rec and bird plans have
// at most one ready move per column and vertical direction, nearly all of
// them at the start; up to side 256 one load of every lane covers a table.
__host__ __device__ inline int sim_cap(int side)
{
    const int c = (side + (side <= 256 ? 63 : 31)) & ~7;
    return side <= 256 && c > 256 ? 256 : c;
}
__host__ __device__ inline int sim_pow2(int side)
{
    int p = 32;
    while (p < side) p <<= 1;
    return p;
}
// Shared memory of a simulation block for grids of at most `side`: the
// tables, the members, the control words, a sort buffer per warp, a list of
// ids, 16 bytes nothing reads, the in-degree counters.
__host__ __device__ inline size_t sim_smem_bytes(int side, int warps, int counters)
{
    const size_t M = (size_t)((side + 7) & ~7);
    return 14 * 4 * (size_t)sim_cap(side) + 12 * M + sizeof(SimCtl) + 4 * ((size_t)sim_pow2(side) * warps + M) + 16 +
           2 * (size_t)((counters + 7) & ~7);
}
constexpr int SIM_MAX_THREADS = 128, SIM_BLOCKS = 16;   // with writers; one-warp blocks per SM

// Workspace of the wide simulation: 8 bytes per move, beside the words per
// vertex that the conflict graph no longer needs. Only instances with more
// ready moves than a shared-memory table holds (at least 64) can need it.
constexpr int SIM_WIDE_MIN = 65;
__host__ __device__ inline size_t sim_wide_bytes(long long k) { return k < SIM_WIDE_MIN ? 0 : 8 * (size_t)k; }

// End of the narrow simulation when an instance needs more table entries
// than shared memory holds: the wide one starts over, in the same block or in
// the kernel that follows (k_sim_wide), so callers never see it.
constexpr int32_t RR_SIM_RETRY = 100;

// A move's record (two int4): the position word of its source; its first
// leg's direction (2 bits) and length (11 bits), its destination row (10
// bits), whether its only successor is the next id, without other
// predecessors (1 bit), and which of the first four successors the next id is
// (3 bits, 0: none); its number of successors; where those after the fourth lie;
// then the first four successors. The position of a token that moves in direction d: the
// coordinate along its way, mirrored for the negative directions so that it
// grows, and the one across it, both plus one, in the halves of a word.
constexpr int MIRROR = 1025;
constexpr int MULTI_BITS = 11, MULTI_COUNT = (1 << MULTI_BITS) - 1;   // a path has at most 2 047 predecessors
__device__ __forceinline__ uint32_t dir_pos(int d, int row, int col)
{
    const int x = d < 2 ? row : col, al = (d & 1) ? x + 1 : MIRROR - 1 - x;
    return (uint32_t)al | (uint32_t)((d < 2 ? col : row) + 1) << 16;
}
__device__ __forceinline__ int4 move_rec(rr_move p, int nsucc, int more, bool chain, int next)
{
    const int hl = p.dst_col - p.src_col, vl = p.dst_row - p.src_row;
    const int d = hl ? (hl > 0 ? 3 : 2) : (vl > 0 ? 1 : 0), len = hl ? (hl > 0 ? hl : -hl) : (vl > 0 ? vl : -vl);
    return make_int4((int)dir_pos(d, p.src_row, p.src_col), d | len << 2 | p.dst_row << 13 | (chain ? 1 << 23 : 0) | next << 24,
                     nsucc, more);
}

// Successor entries carry this flag when the successor has a single
// predecessor: it becomes ready as soon as that predecessor finishes. Other
// entries hold the number of the successor's in-degree counter.
constexpr int32_t SUCC_SINGLE = 1 << 30;
constexpr int32_t SUCC_ID = SUCC_SINGLE - 1;

__device__ __forceinline__ void *arena_alloc(const Arena &A, unsigned long long bytes, bool *ok)
{
    bytes = (bytes + 255ull) & ~255ull;
    unsigned long long off = atomicAdd(A.top, bytes);
    if (off + bytes > A.size) { *ok = false; return nullptr; }
    return A.base + off;
}

__host__ __device__ constexpr unsigned long long arena_pad(unsigned long long bytes) { return (bytes + 255ull) & ~255ull; }

// The lane, read once: threadIdx.x would be read again (20 cycles or more)
// wherever the compiler is short of a register to keep it in.
__device__ __forceinline__ int lane_id()
{
    int l;
    asm volatile("mov.u32 %0, %%laneid;" : "=r"(l));
    return l;
}

__device__ __forceinline__ int warp_incl_scan(int v)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int u = __shfl_up_sync(FULL, v, o);
        if (lane >= o) v += u;
    }
    return v;
}

__device__ __forceinline__ int warp_sum(int v) { return __reduce_add_sync(FULL, v); }

// Bits of rows [lo, hi) that fall in word w (rows 32w .. 32w+31).
__device__ __forceinline__ uint32_t row_mask(int w, int lo, int hi)
{
    int a = max(lo - 32 * w, 0), b = min(hi - 32 * w, 32);
    if (b <= a) return 0u;
    uint32_t hiMask = b >= 32 ? FULL : ((1u << b) - 1u);
    uint32_t loMask = (1u << a) - 1u;
    return hiMask & ~loMask;
}

__device__ __forceinline__ int iabs(int v) { return v < 0 ? -v : v; }

// A move of a list in one 16-byte access where the list is aligned for it
// (an array of rr_move need not be): four 4-byte accesses of a warp's moves
// touch each of their sectors four times.
__device__ __forceinline__ rr_move load_move(const rr_move *p)
{
    if (((uintptr_t)p & 15) == 0) {
        const int4 v = *reinterpret_cast<const int4 *>(p);
        return rr_move{v.x, v.y, v.z, v.w};
    }
    return *p;
}
__device__ __forceinline__ void store_move(rr_move *p, int sr, int sc, int dr, int dc)
{
    if (((uintptr_t)p & 15) == 0) *reinterpret_cast<int4 *>(p) = make_int4(sr, sc, dr, dc);
    else *p = rr_move{sr, sc, dr, dc};
}

// Bring the 32 bytes around a word into L1 without a register waiting for
// them (lanes that c holds for): an asynchronous copy of the word to a place
// in shared memory that nothing reads, `dump`. (prefetch.global.L1 stops at
// L2 here: a load after it takes 300 to 500 cycles, after this copy 40.)
__device__ __forceinline__ uint32_t sh_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void touch_if(bool c, const void *p, uint32_t dump)
{
    asm volatile("{ .reg .pred q; setp.ne.u32 q, %0, 0; @q cp.async.ca.shared.global [%1], [%2], 4; }"
                 ::"r"((unsigned)c), "r"(dump), "l"(p) : "memory");
}
__device__ __forceinline__ void touch_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Test hook: when positive, the pairing loop and the batching simulation
// stop after this many iterations with RR_ERR_TIMEOUT, as when their own
// bounds run out (rr_debug_guard_limit sets it in every module that runs
// them). Zero keeps the built-in bounds.
static __device__ long long g_guard_cap = 0;

// Status helpers: an instance is live while its status is RR_OK.
__device__ __forceinline__ void set_status(rr_instance *I, int st)
{
    atomicCAS(&I->status, 0, st);
}
__device__ __forceinline__ bool live(const rr_instance *I) { return I->status == RR_OK; }

// Adds a warp's elementary-step count to the instance total (every lane of
// the warp calls it).
__device__ __forceinline__ void add_steps(rr_instance *I, long long v)
{
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
    if ((threadIdx.x & 31) == 0 && v) atomicAdd((unsigned long long *)&I->n_steps, (unsigned long long)v);
}

// Largest a in [lo, hi] with a == lo or delta(a) <= 0, for a non-decreasing
// delta (the discrete derivative of a convex cost). Warp-cooperative: every
// round probes 32 evenly spaced candidates.
template <class F>
__device__ int split_search(int lo, int hi, F delta)
{
    const int lane = threadIdx.x & 31;
    for (int guard = 0; hi > lo && guard < 8; ++guard) {
        const int span = hi - lo;
        const int al = lo + (int)(((long long)(lane + 1) * span + 31) / 32);
        const bool ok = delta(al) <= 0;
        const unsigned bal = __ballot_sync(FULL, ok);
        if (bal == 0u) {
            hi = __shfl_sync(FULL, al, 0) - 1;
        } else {
            const int L = 31 - __clz(bal);
            const int aL = __shfl_sync(FULL, al, L);
            const int aN = __shfl_sync(FULL, al, L < 31 ? L + 1 : 31);
            lo = aL;
            if (L < 31) hi = aN - 1;
        }
    }
    return lo;
}

// Number of band atoms i of a target column with (b_i - i) <= T, i.e. with at
// most T - r0 empty band traps above them. hr: the column's band holes.
__device__ __forceinline__ int band_P(const int16_t *hr, int nh, int nband, int r0, int T)
{
    const int u = T - r0;
    if (u < 0) return 0;
    if (u >= nh) return nband;
    return (int)hr[u] - r0 - u;
}

// Shared memory of the bird stage, in words: reservoir-row bits of the largest
// grid (column-major, an odd number of words per column), the two sides' layer
// entries (a side holds fewer than the tokens it needs and one layer more, and
// three words of padding), the two token lists and layer counts, then five
// int16 arrays (the
// receiver list: columns, band atoms, atoms above the band; the current
// receiver's band holes and band atom rows).
constexpr int BIRD_MAX_THREADS = 1024;
struct BirdLayout {
    int keys, room, lists, hist, recv, words;
    __host__ __device__ explicit BirdLayout(int max_side)
    {
        keys = (max_side * (((max_side + 31) / 32) | 1) + 3) & ~3;     // 16-byte aligned, as a side's room is
        room = (2 * max_side + 6) & ~3;
        lists = keys + 2 * room;
        hist = lists + 2 * max_side;
        recv = hist + 4 * max_side;
        words = recv + (5 * max_side + 1) / 2;
    }
};
inline size_t bird_smem_bytes(int max_side) { return 4 * (size_t)BirdLayout(max_side).words; }

} // namespace rrk

// Library-internal hooks between translation units (not part of the C ABI).
int rr_internal_reserve(rr_ctx *ctx, int count);

namespace rrk {
// Per-module setters of g_guard_cap (rr_plan.cu, rr_batch.cu, rr_one.cu).
int guard_cap_plan(long long cap);
int guard_cap_batch(long long cap);
int guard_cap_one(long long cap);
// The single-grid kernel (rr_one.cu): one block of ONE_THREADS threads runs
// planning, Gamma and batching of one grid with sides up to ONE_MAX_SIDE.
constexpr int ONE_THREADS = 256;
constexpr int ONE_MAX_SIDE = 256;
size_t one_smem_bytes(int side, int flags);
const void *one_kernel();
int one_launch(rr_instance h, rr_instance *d_inst, JobWS *d_ws, Arena A, int flags, int side, size_t smem,
               rr_instance *hostOut, cudaStream_t s);
} // namespace rrk
