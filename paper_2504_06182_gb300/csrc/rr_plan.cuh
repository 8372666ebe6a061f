// rr_plan.cuh -- planning stages of the improved red-rec algorithm
// (arXiv 2504.06182, Alg. 1; Sec. III.A exact 1D, Sec. III.C redistribution,
// Sec. III.D parallel ordering: every column of non-negative surplus is
// solved up front, then the donor/receiver pairs are identified by one warp
// and the receivers are solved in parallel).
//
// Every stage takes the whole instance array; B.y selects the instance
// (B.x for the stages that run one block per instance). An instance whose
// status is not RR_OK is skipped.
#pragma once
#include "rr_internal.cuh"

namespace rrk {

// ------------------------------------------------------------ validation

__device__ inline void s_plan_setup(const Blk B, rr_instance *inst, JobWS *wsv, int count, int max_side, Arena A)
{
    const int q = B.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
    rr_instance *I = &inst[q];
    int m = 0, n = 0, h = 0, tw = 0;
    if (q < count) {
        I->n_moves = 0; I->n_steps = 0; I->n_ops = 0; I->n_members = 0;
        if (q == 0) wsv[0].npending = wsv[0].nlacking = 0;
        m = I->m; n = I->n;
        const rr_rect R = I->rect;
        const bool bad = m < 1 || n < 1 || m > max_side || n > max_side || m > RR_MAX_SIDE || n > RR_MAX_SIDE ||
                         R.r0 < 0 || R.r0 >= R.r1 || R.r1 > m || R.c0 < 0 || R.c0 >= R.c1 || R.c1 > n || !I->grid ||
                         (I->layout != RR_U8 && I->layout != RR_BITS32) || I->cap_moves < 0 ||
                         (I->cap_moves > 0 && !I->moves);
        I->status = bad ? RR_ERR_ARG : RR_OK;
        h = R.r1 - R.r0;
        tw = R.c1 - R.c0;
        if (bad) m = n = h = tw = 0;
    }
    // one request to the arena per warp: its instances' sizes, scanned (an
    // atomic per array and instance on the one bump pointer took 82 us for
    // 16 384 chains, this 11 us)
    const int W = (m + 31) >> 5;
    const unsigned long long sz[7] = {
        arena_pad(sizeof(uint32_t) * (unsigned long long)n * W), arena_pad(sizeof(int16_t) * (unsigned long long)n * m),
        arena_pad(sizeof(int16_t) * (unsigned long long)tw * h), arena_pad(sizeof(ColInfo) * (unsigned long long)n),
        arena_pad(sizeof(RecvInfo) * (unsigned long long)n), n ? arena_pad(sizeof(Event) * (unsigned long long)(n + 1)) : 0,
        n ? arena_pad(sizeof(int32_t) * (unsigned long long)(2 * n + 1)) : 0};
    unsigned long long need = 0;
#pragma unroll
    for (int u = 0; u < 7; ++u) need += sz[u];
    unsigned long long incl = need;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long v = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += v;
    }
    unsigned long long off = 0;
    if (lane == 31 && incl) off = atomicAdd(A.top, incl);
    off = __shfl_sync(FULL, off, 31) + incl - need;
    if (n == 0) return;
    JobWS &ws = wsv[q];
    ws.nrecv = 0; ws.nev = 0;
    if (off + need > A.size) { I->status = RR_ERR_WORKSPACE; return; }
    char *at = A.base + off;
    ws.colbits = (uint32_t *)at; at += sz[0];
    ws.atomRows = (int16_t *)at; at += sz[1];
    ws.holeRows = (int16_t *)at; at += sz[2];
    ws.col = (ColInfo *)at; at += sz[3];
    ws.recv = (RecvInfo *)at; at += sz[4];
    ws.ev = (Event *)at; at += sz[5];
    ws.unitOff = (int32_t *)at;
}

// ------------------------------------------------- S0: load and transpose
// Column-major bit columns: word w of column c holds rows 32w .. 32w+31.
// bits32 input, rows 16-byte aligned (a row length of a multiple of 128
// columns and an aligned grid): a warp takes 32 rows x 128 columns, lane l
// reads four words of row 32w + l in one 16-byte load, and each of the four
// 32x32 bit tiles is transposed with 32 ballots. Other rows: a warp takes
// one 32x32 tile, one word per lane.
// u8 input, rows 4-byte aligned: a warp takes 32 rows x 128 columns, lane l
// reads four consecutive bytes (columns 4l .. 4l+3) of each row in one
// 4-byte load, so that a warp reads 128 contiguous bytes per row, and builds
// its four columns' words. Other rows: lane l reads column 32g + l byte by
// byte (32 contiguous bytes per row and warp). Grids of at most NARROW
// columns leave most of those lanes idle: there the lanes take rows, and a vote
// makes a word (16 384 chains of 1 024 traps, before chains on 16-byte
// boundaries had a load of their own, in 36 us instead of 246).
constexpr int NARROW = 8;
__device__ inline void s_transpose(const Blk B, rr_instance *inst, JobWS *wsv, int count)
{
    const int q = B.y;
    if (q >= count) return;
    const rr_instance *I = &inst[q];
    if (!live(I)) return;
    JobWS &ws = wsv[q];
    const int m = I->m, n = I->n, W = (m + 31) >> 5, G = (n + 31) >> 5, G4 = (n + 127) >> 7;
    const int lane = threadIdx.x & 31;
    const int w0 = B.w, nw = B.nw;
    if (I->layout == RR_U8 && n == 1 && ((uintptr_t)I->grid & 15) == 0) {
        // one column: 16 rows per lane and load, both of a lane's loads in
        // flight; half a word each, put together in the even lanes (by votes,
        // four loads of 32 rows at a time: 36 us for 16 384 chains of 1024
        // traps, this 17)
        if (w0 != 0) return;
        const uint8_t *src = (const uint8_t *)I->grid;
        uint4 v[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int row = 16 * (lane + 32 * u);
            v[u] = make_uint4(0u, 0u, 0u, 0u);
            if (row + 16 <= m) v[u] = *reinterpret_cast<const uint4 *>(src + row);
            else
                for (int i = 0; row + i < m; ++i) {
                    const uint32_t b = (uint32_t)src[row + i] << (8 * (i & 3));
                    v[u].x |= i < 4 ? b : 0u;
                    v[u].y |= i >> 2 == 1 ? b : 0u;
                    v[u].z |= i >> 2 == 2 ? b : 0u;
                    v[u].w |= i >> 2 == 3 ? b : 0u;
                }
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            // a byte's lowest bit says whether it is not zero; the product
            // brings the four of a word together in bits 24 to 27
            auto nibble = [](uint32_t x) { return ((__vcmpne4(x, 0u) & 0x01010101u) * 0x01020408u) >> 24 & 15u; };
            const uint32_t half = nibble(v[u].x) | nibble(v[u].y) << 4 | nibble(v[u].z) << 8 | nibble(v[u].w) << 12;
            const uint32_t next = __shfl_down_sync(FULL, half, 1);
            const int w = (lane >> 1) + 16 * u;
            if ((lane & 1) == 0 && w < W) ws.colbits[w] = half | next << 16;
        }
    } else if (I->layout == RR_U8 && n <= NARROW) {
        // a few columns: 32 rows per lane group and load, one vote per word
        // and column, four words at a time
        const uint8_t *src = (const uint8_t *)I->grid;
        for (int item = w0; item < (W + 3) >> 2; item += nw) {
            const int w = 4 * item;
            uint32_t keep[4] = {0u, 0u, 0u, 0u};
            for (int c = 0; c < n; ++c) {
                int x[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int row = 32 * (w + u) + lane;
                    x[u] = row < m ? src[(size_t)row * n + c] : 0;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const uint32_t b = __ballot_sync(FULL, x[u] != 0);
                    if (lane == c) keep[u] = b;
                }
            }
            if (lane < n)
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (w + u < W) ws.colbits[(size_t)lane * W + w + u] = keep[u];
        }
    } else if (I->layout == RR_BITS32) {
        const uint32_t *src = (const uint32_t *)I->grid;
        if ((G & 3) == 0 && ((uintptr_t)src & 15) == 0) {
            for (int item = w0; item < G4 * W; item += nw) {
                const int g4 = item / W, w = item % W;
                const int row = 32 * w + lane;
                uint4 v = make_uint4(0u, 0u, 0u, 0u);
                if (row < m) v = *reinterpret_cast<const uint4 *>(src + (size_t)row * G + 4 * g4);
                const uint32_t x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    uint32_t mine = 0;
#pragma unroll
                    for (int bt = 0; bt < 32; ++bt) {
                        const uint32_t bal = __ballot_sync(FULL, (x[c] >> bt) & 1u);
                        if (bt == lane) mine = bal;
                    }
                    const int col = 32 * (4 * g4 + c) + lane;
                    if (col < n) ws.colbits[(size_t)col * W + w] = mine;
                }
            }
        } else {
            for (int item = w0; item < G * W; item += nw) {
                const int g = item / W, w = item % W;
                const int row = 32 * w + lane;
                const uint32_t x = row < m ? src[(size_t)row * G + g] : 0u;
                uint32_t mine = 0;
#pragma unroll
                for (int bt = 0; bt < 32; ++bt) {
                    const uint32_t bal = __ballot_sync(FULL, (x >> bt) & 1u);
                    if (bt == lane) mine = bal;
                }
                const int col = 32 * g + lane;
                if (col < n) ws.colbits[(size_t)col * W + w] = mine;
            }
        }
    } else {
        const uint8_t *src = (const uint8_t *)I->grid;
        if ((n & 3) == 0 && ((uintptr_t)src & 3) == 0) {
            for (int item = w0; item < G4 * W; item += nw) {
                const int g4 = item / W, w = item % W;
                const int c0 = 128 * g4 + 4 * lane;
                if (c0 >= n) continue;
                const int rmax = min(32, m - 32 * w);
                const uint8_t *rp = src + (size_t)(32 * w) * n + c0;
                uint32_t a0 = 0u, a1 = 0u, a2 = 0u, a3 = 0u;
                for (int r = 0; r < rmax; ++r) {
                    const uint32_t v = *reinterpret_cast<const uint32_t *>(rp + (size_t)r * n);
                    a0 |= (uint32_t)((v & 0xffu) != 0u) << r;
                    a1 |= (uint32_t)((v & 0xff00u) != 0u) << r;
                    a2 |= (uint32_t)((v & 0xff0000u) != 0u) << r;
                    a3 |= (uint32_t)((v & 0xff000000u) != 0u) << r;
                }
                uint32_t *out = ws.colbits + (size_t)c0 * W + w;
                out[0] = a0;
                out[W] = a1;
                out[2 * W] = a2;
                out[3 * W] = a3;
            }
        } else {
            for (int item = w0; item < G * W; item += nw) {
                const int g = item / W, w = item % W;
                const int col = 32 * g + lane;
                if (col >= n) continue;
                const int rmax = min(32, m - 32 * w);
                uint32_t mine = 0;
                for (int r = 0; r < rmax; ++r) mine |= (uint32_t)(src[(size_t)(32 * w + r) * n + col] != 0) << r;
                ws.colbits[(size_t)col * W + w] = mine;
            }
        }
    }
}

// -------------------------------------- S1-S3: counts, surplus, column solves
// One warp per column. Target columns of non-negative surplus get the exact
// 1D solve: the h sources are the band atoms plus the a nearest atoms above
// and the x-a nearest below (a contiguous window of the sorted sources),
// a chosen by minimum total distance with the largest a on ties. Columns
// outside the target columns are pushed into their reservoir rows when they
// have the atoms for it, unless `strict` (then only their reservoir-row atoms
// are donatable and nothing in them moves).
__device__ inline void s_colstats(const Blk B, rr_instance *inst, JobWS *wsv, int count, int strict)
{
    const int q = B.y;
    if (q >= count) return;
    const rr_instance *I = &inst[q];
    if (!live(I)) return;
    JobWS &ws = wsv[q];
    const int m = I->m, n = I->n, W = (m + 31) >> 5;
    const int r0 = I->rect.r0, r1 = I->rect.r1, c0 = I->rect.c0, c1 = I->rect.c1;
    const int h = r1 - r0, R = m - h;
    const int lane = threadIdx.x & 31;
    for (int c = B.w; c < n; c += B.nw) {
        const uint32_t x = lane < W ? ws.colbits[(size_t)c * W + lane] : 0u;
        const uint32_t mT = row_mask(lane, 0, r0), mBd = row_mask(lane, r0, r1), mO = row_mask(lane, r1, m);
        const int K = warp_sum(__popc(x));
        const int ntop = warp_sum(__popc(x & mT));
        const int nband = warp_sum(__popc(x & mBd));
        const int nbot = warp_sum(__popc(x & mO));
        int16_t *rows = ws.atomRows + (size_t)c * m;
        const bool target = c >= c0 && c < c1;
        int16_t *hr = target ? ws.holeRows + (size_t)(c - c0) * h : nullptr;
        // the atoms' rows, and a target column's band holes: a word at a time,
        // a row per lane, so that a store covers consecutive places (a word
        // per lane and its bits in turn: 241 us for 2 000 grids of sides 33
        // to 251, this 116 us)
        int pa = 0, ph = 0;
        const unsigned lt = (1u << lane) - 1u;
        for (int w = 0; w < W; ++w) {
            const uint32_t xw = __shfl_sync(FULL, x, w);
            if ((xw >> lane) & 1u) rows[pa + __popc(xw & lt)] = (int16_t)(32 * w + lane);
            pa += __popc(xw);
            if (target) {
                const uint32_t hw = ~xw & row_mask(w, r0, r1);
                if ((hw >> lane) & 1u) hr[ph + __popc(hw & lt)] = (int16_t)(32 * w + lane);
                ph += __popc(hw);
            }
        }
        __syncwarp();

        ColInfo ci;
        ci.K = K; ci.ntop = ntop; ci.nband = nband; ci.nbot = nbot;
        ci.a = 0; ci.kd_end = 0; ci.ku_start = 0; ci.nmoves = 0; ci.topRun = 0; ci.botRun = 0;
        ci.tbase = 0; ci.bbase = 0;
        if (target) {
            ci.sigma = K - h;
            if (ci.sigma >= 0) {
                ci.kind = KIND_TARGET_SOLVED;
                const int need = h - nband, nh = h - nband;
                const int lo = max(0, need - nbot), hi = min(need, ntop);
                // d cost/da = (r0+a-1 - top(a-1)) + (2 P(r0+a-1) - M) + (r0+h-need+a-1 - bot(need-a))
                const int a = split_search(lo, hi, [&](int aa) {
                    const int topRow = rows[ntop - aa];                  // (aa-1)-th nearest above
                    const int botRow = rows[ntop + nband + (need - aa)]; // (need-aa)-th nearest below
                    return (r0 + aa - 1 - topRow) + (2 * band_P(hr, nh, nband, r0, r0 + aa - 1) - nband) +
                           (r0 + h - need + aa - 1 - botRow);
                });
                ci.a = a;
                ci.kd_end = a + band_P(hr, nh, nband, r0, r0 + a - 1);
                ci.ku_start = a + band_P(hr, nh, nband, r0, r0 + a);
                ci.nmoves = ci.kd_end + (h - ci.ku_start);
                ci.ptop = ntop - a;
                ci.pbot = nbot - (need - a);
                ci.tbase = ntop - a - 1;
                ci.bbase = ntop - a + h;
            } else {
                ci.kind = KIND_RECEIVER;
                ci.ptop = 0; ci.pbot = 0;
            }
        } else if (!strict && K >= R) {
            // Virtual targets = this column's reservoir cells: the first r0
            // atoms go to rows 0..r0-1, the last m-r1 to rows r1..m-1.
            ci.kind = KIND_OUTER_FULL;
            ci.sigma = R; ci.ptop = r0; ci.pbot = m - r1;
            const uint32_t valid = row_mask(lane, 0, m);
            const uint32_t brk = ~x | ~valid;                     // first non-atom from row 0
            const int fz = brk ? 32 * lane + __ffs(brk) - 1 : 0x7fffffff;
            int firstZero = fz;
            firstZero = __reduce_min_sync(FULL, firstZero);
            if (firstZero > m) firstZero = m;
            const uint32_t z2 = ~x & valid;                       // last empty row
            int lz = z2 ? 32 * lane + 31 - __clz(z2) : -1;
            lz = __reduce_max_sync(FULL, lz);
            ci.topRun = min(firstZero, r0);
            ci.botRun = min(m - 1 - lz, m - r1);
            ci.nmoves = (r0 - ci.topRun) + (m - r1 - ci.botRun);
        } else {
            ci.kind = KIND_OUTER_PART;
            ci.sigma = ntop + nbot; ci.ptop = ntop; ci.pbot = nbot;
            ci.tbase = ntop - 1; ci.bbase = ntop + nband;
        }
        if (lane == 0) ws.col[c] = ci;
    }
}

// ------------------------------------------------- S4: pairing (one warp)

constexpr size_t WARM_BYTES = 160 * 1024;    // rows that fit L1 beside the pairing's shared memory

// What the pairing keeps of a column in shared memory.
struct PairCol {
    int16_t kind, ptop, pbot, tbase, bbase, nband;   // as in ColInfo
    int16_t tT, bT;          // donor: pool cursors
    int16_t mandT, mandB;    // receiver: atoms above / below the band so far
    int16_t nev, recv;       // receiver: its events, its place in saturation order
};
// (rr_capi.cu, rr_noalloc.cu and the single-grid kernel size it by this, 64
// bytes more)
static_assert(sizeof(PairCol) == 24 && PAIR_BYTES == 8 + 4 + 24 + 3 * 2, "shared memory of the pairing");

// Score of the pair of columns c < v with surpluses s1 and s2 (v < 0: none).
// Larger is better: tokens exchanged, then smaller gap, then smaller deficit,
// then smaller receiver index, then smaller donor index; c last.
__device__ __forceinline__ uint2 pair_score(int c, int v, int s1, int s2)
{
    const bool right = s1 > 0;                        // the donor is c
    const int give = right ? s1 : s2, need = -(right ? s2 : s1), j = right ? v : c;
    uint2 r;
    r.y = (unsigned)min(give, need) << 10 | (unsigned)(1023 - (v - c));
    r.x = (unsigned)(2047 - need) << 21 | (unsigned)(1023 - j) << 11 | (right ? 1u << 10 : 0u) | (unsigned)c;
    const bool none = v < 0 || s1 == 0 || s2 == 0 || (s1 > 0) == (s2 > 0);
    return none ? make_uint2(0u, 0u) : r;
}

// The pairing loop is one chain: the best pair, the donor's tokens it takes
// (a search over rows in global memory), the scores that change. So each
// column's best-pair score stays in shared memory and the best of a lane's
// columns in its registers (two warp reductions find the pair); at most three
// scores change per pair (its two columns' and that of the column before
// them), computed side by side from values in registers; what is needed of a
// column is in shared memory; and `warm` (calls over few grids) brings the
// atoms' and holes' rows into L1 first. One 256 x 256 grid, 241 pairs: 243 us
// (with the scores rescanned, one lane updating them, and rows from L2: 400).
__device__ inline void s_pair(const Blk B, rr_instance *inst, JobWS *wsv, int count, int warm)
{
    extern __shared__ unsigned long long smem_u64[];
    const int q = B.x;
    if (q >= count) return;
    rr_instance *I = &inst[q];
    if (!live(I)) return;
    JobWS &ws = wsv[q];
    const int m = I->m, n = I->n;
    const int r0 = I->rect.r0, r1 = I->rect.r1, c0 = I->rect.c0;
    const int h = r1 - r0;
    const int lane = threadIdx.x & 31;

    uint2 *score = (uint2 *)smem_u64;                 // n: of the pair of a column and the next one in the list
    int32_t *sig = (int32_t *)(smem_u64 + n);         // n: surplus
    PairCol *col = (PairCol *)(sig + n);
    int16_t *prv = (int16_t *)(col + n), *nxt = prv + n, *evOrd = nxt + n;
    const uint32_t dump = sh_addr((void *)(((uintptr_t)(evOrd + n) + 15) & ~(uintptr_t)15));
    if (warm) {
        const size_t ba = 2 * (size_t)n * m, bh = 2 * (size_t)(I->rect.c1 - c0) * h;
        if (ba + bh <= WARM_BYTES) {
            for (size_t o = 32 * (size_t)lane; o < ba; o += 1024) touch_if(true, (const char *)ws.atomRows + o, dump);
            for (size_t o = 32 * (size_t)lane; o < bh; o += 1024) touch_if(true, (const char *)ws.holeRows + o, dump);
        }
    }

    int tot = 0, nneg = 0;
    for (int c = lane; c < n; c += 32) {
        const ColInfo ci = ws.col[c];
        sig[c] = ci.sigma;
        col[c] = PairCol{(int16_t)ci.kind, (int16_t)ci.ptop, (int16_t)ci.pbot, (int16_t)ci.tbase, (int16_t)ci.bbase,
                         (int16_t)ci.nband, 0, 0, (int16_t)ci.ntop, (int16_t)ci.nbot, 0, -1};
        tot += ci.sigma;
        nneg += ci.sigma < 0;
    }
    tot = warp_sum(tot);
    nneg = warp_sum(nneg);
    touch_wait();
    if (tot < 0) {                    // some column can never be saturated (Sec. III.C)
        if (lane == 0) { I->status = RR_INFEASIBLE; I->n_moves = 0; }
        return;
    }
    __syncwarp();
    // list of non-zero-surplus columns: next (right-to-left sweep) and prev
    {
        int carry = -1;
        for (int base = ((n - 1) >> 5) << 5; base >= 0; base -= 32) {
            const int c = base + lane;
            const unsigned nz = __ballot_sync(FULL, c < n && sig[c] != 0);
            const unsigned above = lane < 31 ? nz & ~((2u << lane) - 1u) : 0u;
            if (c < n) nxt[c] = (int16_t)(above ? base + __ffs(above) - 1 : carry);
            if (nz) carry = base + __ffs(nz) - 1;
        }
        carry = -1;
        for (int base = 0; base < n; base += 32) {
            const int c = base + lane;
            const unsigned nz = __ballot_sync(FULL, c < n && sig[c] != 0);
            const unsigned below = nz & ((1u << lane) - 1u);
            if (c < n) prv[c] = (int16_t)(below ? base + 31 - __clz(below) : carry);
            if (nz) carry = base + 31 - __clz(nz);
        }
    }
    __syncwarp();
    for (int c = lane; c < n; c += 32) {
        const int v = nxt[c];
        score[c] = pair_score(c, v, sig[c], v >= 0 ? sig[v] : 0);
    }
    // the best of this lane's columns c = lane, lane + 32, ...
    unsigned mine_y = 0u, mine_x = 0u;
    auto best_of_lane = [&]() {
        mine_y = mine_x = 0u;
#pragma unroll 4
        for (int c = lane; c < n; c += 32) {
            const uint2 s = score[c];
            const bool more = s.y > mine_y || (s.y == mine_y && s.x > mine_x);
            mine_y = more ? s.y : mine_y;
            mine_x = more ? s.x : mine_x;
        }
    };
    best_of_lane();

    int nrecv = 0, nev = 0;
    const int16_t *allRows = ws.atomRows;
    for (int iter = 0; nneg > 0; ++iter) {
        if (iter > n || (g_guard_cap > 0 && iter >= g_guard_cap)) { if (lane == 0) I->status = RR_ERR_TIMEOUT; return; }
        const unsigned by = __reduce_max_sync(FULL, mine_y);
        if (by == 0u) { if (lane == 0) I->status = RR_ERR_INTERNAL; return; }
        const int cl = (int)(__reduce_max_sync(FULL, mine_y == by ? mine_x : 0u) & 1023u);   // the pair: cl and
        const int cr = nxt[cl], pl = prv[cl], nr = nxt[cr];                                   // cr; around it: pl, nr
        const int sl0 = sig[cl], sr0 = sig[cr], spl = pl >= 0 ? sig[pl] : 0, snr = nr >= 0 ? sig[nr] : 0;
        const int i = sl0 > 0 ? cl : cr, j = sl0 > 0 ? cr : cl;
        const int si = sl0 > 0 ? sl0 : sr0, need = -(sl0 > 0 ? sr0 : sl0);
        const int x = min(si, need);
        const int kase = si > need ? 1 : (si == need ? 2 : 3);
        const PairCol D = col[i], Rj = col[j];
        const int16_t *drows = allRows + (size_t)i * m;
        const int t0 = D.tT, b0 = D.bT;
        const int availT = D.ptop - t0, availB = D.pbot - b0;
        const int e = nev++;
        if (e >= n) { if (lane == 0) I->status = RR_ERR_INTERNAL; return; }   // an event settles a column
        int a;
        __syncwarp();
        if (kase == 3) {
            a = availT;
            if (lane == 0) {
                col[j].mandT = (int16_t)(Rj.mandT + availT); col[j].mandB = (int16_t)(Rj.mandB + availB);
                col[i].tT = D.ptop; col[i].bT = D.pbot;
            }
        } else {
            const int mT = Rj.mandT, mB = Rj.mandB;
            const int M = Rj.nband, nh = h - M;
            const int16_t *hr = ws.holeRows + (size_t)(j - c0) * h;
            if (kase == 2) {
                a = availT;
                if (availT + availB != x) { if (lane == 0) I->status = RR_ERR_INTERNAL; return; }
            } else {
                const int lo = max(0, x - availB), hi = min(x, availT);
                const bool full = D.kind == KIND_OUTER_FULL;
                a = split_search(lo, hi, [&](int aa) {
                    const int lt = t0 + aa - 1, lb = b0 + x - aa;      // the donor's next pool atoms
                    const int tr = full ? r0 - 1 - lt : (int)drows[D.tbase - lt];
                    const int br = full ? r1 + lb : (int)drows[D.bbase + lb];
                    return (r0 + mT + aa - 1 - tr) + (2 * band_P(hr, nh, M, r0, r0 + mT + aa - 1) - M) +
                           (r0 + h - mB - x + aa - 1 - br);
                });
            }
            const int nT = mT + a;
            const int kd = nT + band_P(hr, nh, M, r0, r0 + nT - 1), ku = nT + band_P(hr, nh, M, r0, r0 + nT);
            if (lane == 0) {
                col[i].tT = (int16_t)(t0 + a); col[i].bT = (int16_t)(b0 + x - a);
                col[j].recv = (int16_t)nrecv;
                RecvInfo ri;
                ri.j = j;
                ri.ev_first = 0;
                ri.ncontrib = Rj.nev + 1;
                ri.nT = nT;
                ri.kd_end = kd;
                ri.ku_start = ku;
                ri.nmoves = kd + (h - ku);
                ri.pad = 0;
                ws.recv[nrecv] = ri;
            }
            ++nrecv;
            --nneg;
        }
        // surpluses after it, the columns that reached zero out of the list,
        // the three scores that change
        const int sl = sl0 > 0 ? sl0 - x : sl0 + x, sr = sr0 > 0 ? sr0 - x : sr0 + x;
        const bool zl = sl == 0, zr = sr == 0;
        const int afterPl = zl ? (zr ? nr : cr) : cl, sAfterPl = zl ? (zr ? snr : sr) : sl;
        const int afterL = zr ? nr : cr, sAfterL = zr ? snr : sr;
        if (lane == 0) {
            evOrd[e] = Rj.nev;
            col[j].nev = (int16_t)(Rj.nev + 1);
            Event ev;
            ev.kase = kase; ev.i = i; ev.j = j; ev.x = x; ev.a = a; ev.t0 = t0; ev.b0 = b0; ev.at = -1;
            ws.ev[e] = ev;
            sig[cl] = sl;
            sig[cr] = sr;
            if (pl >= 0) nxt[pl] = (int16_t)afterPl;
            if (!zl) nxt[cl] = (int16_t)afterL;
            if (!zr) prv[cr] = (int16_t)(zl ? pl : cl);
            if (nr >= 0) prv[nr] = (int16_t)(zr ? (zl ? pl : cl) : cr);
        }
        {
            const int c = lane == 0 ? pl : lane == 1 ? cl : cr;
            const uint2 s = lane == 0 ? pair_score(pl, afterPl, spl, sAfterPl)
                                      : lane == 1 ? pair_score(cl, afterL, sl, sAfterL) : pair_score(cr, nr, sr, snr);
            if (lane < 3 && c >= 0) score[c] = s;
        }
        __syncwarp();
        if ((pl & 31) == lane || (cl & 31) == lane || (cr & 31) == lane) best_of_lane();
        __syncwarp();
    }
    // the events ordered by receiver: a receiver's first slot, then each
    // event's slot
    for (int base = 0, carry = 0; base < nrecv; base += 32) {
        const int r = base + lane;
        const int v = r < nrecv ? ws.recv[r].ncontrib : 0;
        const int incl = warp_incl_scan(v);
        if (r < nrecv) { ws.recv[r].ev_first = carry + incl - v; sig[r] = carry + incl - v; }
        carry += __shfl_sync(FULL, incl, 31);
    }
    __syncwarp();
    for (int e = lane; e < nev; e += 32) ws.ev[sig[col[ws.ev[e].j].recv] + evOrd[e]].at = e;
    // move offsets of all solve units: column units in column order, then
    // receiver units in saturation order
    int carry = 0;
    const int U = n + nrecv;
    for (int base = 0; base < U; base += 32) {
        const int u = base + lane;
        int v = 0;
        if (u < n) v = ws.col[u].nmoves;
        else if (u < U) v = ws.recv[u - n].nmoves;
        const int incl = warp_incl_scan(v);
        if (u < U) ws.unitOff[u] = carry + incl - v;
        carry += __shfl_sync(FULL, incl, 31);
    }
    if (lane == 0) {
        ws.unitOff[U] = carry;
        ws.nrecv = nrecv;
        ws.nev = nev;
        I->n_moves = carry;
        if ((int64_t)carry > I->cap_moves) I->status = RR_ERR_CAPACITY;
    }
}

// The instances that need no pairing (no column lacks atoms, as in 1D chains,
// or the whole grid does) are done with here, a warp each; the others are
// listed for s_pair. In a call over many grids that leaves s_pair's blocks,
// whose shared memory is sized for the largest side, to those that need it:
// 16 384 chains of 1024 traps, five such blocks per SM, 51 -> 14 us.
__device__ inline void s_pair_sift(const Blk B, rr_instance *inst, JobWS *wsv, int count)
{
    const int lane = threadIdx.x & 31, q = B.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (q >= count) return;
    rr_instance *I = &inst[q];
    if (!live(I)) return;
    JobWS &ws = wsv[q];
    const int n = I->n;
    int tot = 0;
    bool lacks = false;
#pragma unroll 4
    for (int c = lane; c < n; c += 32) {
        const int sigma = ws.col[c].sigma;
        tot += sigma;
        lacks |= sigma < 0;
    }
    tot = warp_sum(tot);
    if (tot < 0) {                    // some column can never be saturated (Sec. III.C)
        if (lane == 0) { I->status = RR_INFEASIBLE; I->n_moves = 0; }
        return;
    }
    if (__any_sync(FULL, lacks)) {
        if (lane == 0) wsv[atomicAdd(&wsv[0].npending, 1)].pending = q;
        return;
    }
    int carry = 0;
    for (int base = 0; base < n; base += 32) {
        const int c = base + lane, v = c < n ? ws.col[c].nmoves : 0, incl = warp_incl_scan(v);
        if (c < n) ws.unitOff[c] = carry + incl - v;
        carry += __shfl_sync(FULL, incl, 31);
    }
    if (lane != 0) return;
    ws.unitOff[n] = carry;
    ws.nrecv = ws.nev = 0;
    I->n_moves = carry;
    if ((int64_t)carry > I->cap_moves) I->status = RR_ERR_CAPACITY;
}

// ------------------------------------------------------ S6: column units

__device__ inline void s_emit_cols(const Blk B, rr_instance *inst, JobWS *wsv, int count)
{
    const int q = B.y;
    if (q >= count) return;
    rr_instance *I = &inst[q];
    if (!live(I)) return;
    JobWS &ws = wsv[q];
    const int m = I->m, n = I->n;
    const int r0 = I->rect.r0, r1 = I->rect.r1, h = r1 - r0;
    const int lane = threadIdx.x & 31;
    rr_move *out = I->moves;
    long long steps = 0;
    for (int c = B.w; c < n; c += B.nw) {
        const ColInfo ci = ws.col[c];
        if (ci.nmoves == 0) continue;
        const int16_t *rows = ws.atomRows + (size_t)c * m;
        rr_move *o = out + ws.unitOff[c];
        if (ci.kind == KIND_TARGET_SOLVED) {
            const int w = ci.ntop - ci.a;
            for (int k0 = lane; k0 < h; k0 += 128) {
                // four loads in flight (each behind the store before it: 49 us
                // for 16 384 chains of 1024 traps; this 39)
                int src[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) src[u] = k0 + 32 * u < h ? rows[w + k0 + 32 * u] : 0;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int k = k0 + 32 * u;
                    const bool down = k < ci.kd_end, up = k >= ci.ku_start && k < h;   // (else isolated)
                    if (!down && !up) continue;
                    // toward larger rows deepest first, then toward smaller rows
                    store_move(&o[down ? ci.kd_end - 1 - k : ci.kd_end + (k - ci.ku_start)], src[u], c, r0 + k, c);
                    steps += iabs(r0 + k - src[u]);
                }
            }
        } else {   // KIND_OUTER_FULL
            const int nbg = m - r1, ndown = nbg - ci.botRun;
            for (int k = lane; k < ndown; k += 32) {
                store_move(&o[ndown - 1 - k], rows[ci.K - nbg + k], c, r1 + k, c);
                steps += r1 + k - rows[ci.K - nbg + k];
            }
            for (int k = ci.topRun + lane; k < r0; k += 32) {
                store_move(&o[ndown + (k - ci.topRun)], rows[k], c, k, c);
                steps += rows[k] - k;
            }
        }
    }
    add_steps(I, steps);
}

// ---------------------------------------------------- S5/S6: receiver units

// A receiver's h sources, 32 at a time, a source per lane. A warp takes a
// whole receiver, or where there are enough warps (single grids) 32 of its
// sources. The receiver's contributors (the donors of its pairing events) are
// read side by side, one per lane; each one's sources become a bit column in
// the warp's part of shared memory (consecutive atoms: the donor's bit column
// between two rows), a lane per word, so that a source's rank takes one load
// and one popcount per contributor. What bounds it is the chain of dependent
// loads before the first rank (receiver, column, events, donors, their rows),
// which a warp goes through once per receiver. 2 000 grids of sides 33 to 251:
// 870 us by a block per receiver with binary searches over the donors' rows,
// 379 with ranks by popcounts over whole bit columns in global memory, 270
// this way.
struct Contrib {
    int32_t col, full;           // donor; an outer column whose reservoir rows are all filled
    int32_t cnt, tCnt, tAt, bAt; // sources, of these above the band, the nearest ones' atom (row, if full)
    int32_t d, right, first;     // distance, right-side donor, first source index
};

constexpr int EMIT_WARPS = 8;    // at most, per block
constexpr int EMIT_GROUP = 16;   // contributors held in shared memory at a time

// A warp's view of a receiver unit: contributors and the bit columns (32
// words) of their sources, the receiver's own bit column, and the number of
// sources in the words before.
struct EmitUnit {
    const rr_instance *I;
    const JobWS *ws;
    Contrib *C;
    uint32_t *X, *own, *before;
    RecvInfo ri;
    int K;                       // own atoms
    long long out;               // first move
};

// Contributors g0 .. g0 + EMIT_GROUP - 1 of a unit, the first one's first
// source being number *first (moved on); returns their sources in this lane's
// word.
__device__ __forceinline__ int emit_load(const EmitUnit &U, int g0, int *first)
{
    const int lane = threadIdx.x & 31, m = U.I->m, r0 = U.I->rect.r0, r1 = U.I->rect.r1, j = U.ri.j;
    const JobWS &ws = *U.ws;
    __syncwarp();
    const bool act = lane < EMIT_GROUP && g0 + lane < U.ri.ncontrib;
    Contrib c;
    c.col = c.full = 0;
    int cnt = 0, tLo = 0, tHi = 0, bLo = 0, bHi = 0;
    if (act) {
        const Event ev = ws.ev[ws.ev[U.ri.ev_first + g0 + lane].at];
        const ColInfo D = ws.col[ev.i];
        const int16_t *drows = ws.atomRows + (size_t)ev.i * m;
        const int tStart = ev.t0, bStart = ev.b0;
        c.tCnt = ev.kase == 3 ? D.ptop - ev.t0 : ev.a;
        cnt = c.tCnt + (ev.kase == 3 ? D.pbot - ev.b0 : ev.x - ev.a);
        c.full = D.kind == KIND_OUTER_FULL;
        c.col = ev.i;
        c.tAt = c.full ? r0 - 1 - tStart : D.tbase - tStart;
        c.bAt = c.full ? r1 + bStart : D.bbase + bStart;
        c.d = iabs(ev.i - j); c.right = ev.i > j;
        // its sources on a side are consecutive atoms of its column
        // (consecutive rows in a filled outer column): the rows they span
        auto row_of = [&](int at) { return c.full ? at : (int)drows[at]; };
        if (c.tCnt > 0) { tLo = row_of(c.tAt - c.tCnt + 1); tHi = row_of(c.tAt) + 1; }
        if (cnt > c.tCnt) { bLo = row_of(c.bAt); bHi = row_of(c.bAt + cnt - c.tCnt - 1) + 1; }
        c.cnt = cnt;
    }
    const int incl = warp_incl_scan(cnt);
    c.first = *first + incl - cnt;
    if (act) U.C[lane] = c;
    *first += __shfl_sync(FULL, incl, 31);
    int held = 0;
    const int some = min(EMIT_GROUP, U.ri.ncontrib - g0), W = (m + 31) >> 5;
    for (int v = 0; v < some; ++v) {
        const int tl = __shfl_sync(FULL, tLo, v), th = __shfl_sync(FULL, tHi, v);
        const int bl = __shfl_sync(FULL, bLo, v), bh = __shfl_sync(FULL, bHi, v);
        const int col = __shfl_sync(FULL, c.col, v), full = __shfl_sync(FULL, c.full, v);
        uint32_t x = row_mask(lane, tl, th) | row_mask(lane, bl, bh);
        if (!full && lane < W) x &= ws.colbits[(size_t)col * W + lane];
        U.X[v * 32 + lane] = x;
        held += __popc(x);
    }
    __syncwarp();
    return held;
}

// In a row above the band the farther column comes first, right before left,
// the receiver's own (distance 0) last; below it the own, then the nearer
// column, left before right. Whether column a comes before column b.
__device__ __forceinline__ bool emit_before(bool top, int da, int ra, int db, int rb)
{
    return top ? da > db || (da == db && ra && !rb) : da < db || (da == db && !ra && rb);
}

// The move of the source of rank k.
__device__ __forceinline__ int emit_store(const EmitUnit &U, rr_instance *I, int k, int row, int col)
{
    const int h = I->rect.r1 - I->rect.r0, r0 = I->rect.r0;
    const int pos = k < U.ri.kd_end ? U.ri.kd_end - 1 - k : U.ri.kd_end + (k - U.ri.ku_start);
    if (k < 0 || k >= h || pos >= U.ri.nmoves) {
        set_status(I, RR_ERR_INTERNAL);
        return 0;
    }
    if (pos < U.ri.kd_end && k >= U.ri.kd_end) return 0;             // isolated own band atom
    store_move(&I->moves[U.out + pos], row, col, r0 + k, U.ri.j);
    return iabs(r0 + k - row) + iabs(U.ri.j - col);
}

// A unit of more contributors than shared memory holds: its sources 32 at a
// time, whichever contributors they come from, all contributors read in turn
// for each 32. part of parts: the 32s that this warp takes.
static __device__ __noinline__ int emit_many(const EmitUnit U, rr_instance *I, int part, int parts)
{
    const int lane = threadIdx.x & 31, h = I->rect.r1 - I->rect.r0, r0 = I->rect.r0, nc = U.ri.ncontrib;
    const int16_t *atomRows = U.ws->atomRows;
    int steps = 0;
    for (int t0 = 32 * part; t0 < h; t0 += 32 * parts) {
        const int t = t0 + lane;
        int row = t < U.K && t < h ? atomRows[(size_t)U.ri.j * I->m + t] : 0, col = U.ri.j, ci = -1, sd = 0, sr = 0;
        for (int g0 = 0, first = U.K; g0 < nc; g0 += EMIT_GROUP) {
            const int before = first;
            emit_load(U, g0, &first);
            if (t >= before && t < first) {
                int lo = 0, hi = min(EMIT_GROUP, nc - g0) - 1;       // contributor holding source t
                while (lo < hi) { const int mid = (lo + hi + 1) >> 1; if (U.C[mid].first <= t) lo = mid; else hi = mid - 1; }
                const Contrib c = U.C[lo];
                const int u = t - c.first, at = u < c.tCnt ? c.tAt - u : c.bAt + (u - c.tCnt);
                ci = g0 + lo; sd = c.d; sr = c.right; col = c.col;
                row = c.full ? at : atomRows[(size_t)col * I->m + at];
            }
        }
        const int w = row >> 5;
        const uint32_t bit = 1u << (row & 31);
        const bool top = row < r0;
        int k = (int)U.before[w] + __popc(U.own[w] & (bit - 1u));
        if (ci >= 0 && !top && (U.own[w] & bit)) ++k;
        for (int g0 = 0, first = U.K; g0 < nc; g0 += EMIT_GROUP) {
            emit_load(U, g0, &first);
            for (int v = 0; v < min(EMIT_GROUP, nc - g0); ++v) {
                const uint32_t x = U.X[v * 32 + w];
                k += __popc(x & (bit - 1u));
                if ((x & bit) && g0 + v != ci) k += emit_before(top, U.C[v].d, U.C[v].right, sd, sr);
            }
        }
        if (t < h) steps += emit_store(U, I, k, row, col);
    }
    return steps;
}

__device__ inline void s_emit_recv(const Blk B, rr_instance *inst, JobWS *wsv, int count)
{
    __shared__ Contrib Call[EMIT_WARPS][EMIT_GROUP];
    __shared__ uint32_t Xall[EMIT_WARPS][(EMIT_GROUP + 2) * 32];
    const int q = B.y;
    if (q >= count) return;
    rr_instance *I = &inst[q];
    if (!live(I)) return;
    JobWS &ws = wsv[q];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int m = I->m, n = I->n, r0 = I->rect.r0, h = I->rect.r1 - r0;
    const int W = (m + 31) >> 5, chunks = (h + 31) >> 5;
    const int split = B.nw >= ws.nrecv * chunks ? chunks : 1, items = ws.nrecv * split;
    EmitUnit U;
    U.I = I; U.ws = &ws; U.C = Call[wid]; U.X = Xall[wid]; U.own = U.X + EMIT_GROUP * 32; U.before = U.own + 32;
    long long steps = 0;
    for (int it = B.w; it < items; it += B.nw) {
        const int r = it / split, part = it - r * split;
        U.ri = ws.recv[r];
        const int j = U.ri.j, nc = U.ri.ncontrib;
        const uint32_t mine = lane < W ? ws.colbits[(size_t)j * W + lane] : 0u;
        U.K = ws.col[j].K;
        U.out = ws.unitOff[n + r];
        int first = U.K, held = __popc(mine);
        __syncwarp();
        U.own[lane] = mine;
        for (int g0 = 0; g0 < nc; g0 += EMIT_GROUP) held += emit_load(U, g0, &first);
        U.before[lane] = (uint32_t)(warp_incl_scan(held) - held);
        __syncwarp();
        if (first != h) {
            if (lane == 0) set_status(I, RR_ERR_INTERNAL);
            continue;
        }
        if (nc > EMIT_GROUP) {
            steps += emit_many(U, I, part, split);
            continue;
        }
        // the own atoms: a source's rank is the number of sources in rows
        // below it and, in its own row, of those that come first
        const int16_t *own = ws.atomRows + (size_t)j * m;
        for (int t = 32 * part + lane; t < U.K; t += 32 * split) {
            const int row = own[t], w = row >> 5;
            const uint32_t bit = 1u << (row & 31), upto = row < r0 ? bit | (bit - 1u) : bit - 1u;
            int k = (int)U.before[w] + __popc(U.own[w] & (bit - 1u));
            for (int v = 0; v < nc; ++v) k += __popc(U.X[v * 32 + w] & upto);
            steps += emit_store(U, I, k, row, j);
        }
        // each contributor's
        for (int c = part; c < nc; c += split) {
            const Contrib D = U.C[c];
            const int16_t *rows = ws.atomRows + (size_t)D.col * m;
            for (int u = lane; u < D.cnt; u += 32) {
                const int at = u < D.tCnt ? D.tAt - u : D.bAt + (u - D.tCnt);
                const int row = D.full ? at : rows[at], w = row >> 5;
                const bool top = row < r0;
                const uint32_t bit = 1u << (row & 31);
                int k = (int)U.before[w] + __popc(U.own[w] & (top ? bit - 1u : bit | (bit - 1u)));
                for (int v = 0; v < nc; ++v) {
                    const uint32_t x = U.X[v * 32 + w];
                    k += __popc(x & (bit - 1u));
                    if ((x & bit) && v != c) k += emit_before(top, U.C[v].d, U.C[v].right, D.d, D.right);
                }
                steps += emit_store(U, I, k, row, D.col);
            }
        }
    }
    add_steps(I, steps);
}

} // namespace rrk
