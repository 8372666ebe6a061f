// rr_bird.cuh -- planning stage of the bird algorithm (arXiv 2504.06182,
// Alg. 2, Sec. III.E).
//
// The column phase is red-rec's (k_colstats and k_emit_cols: every column of
// non-negative surplus solved by the exact 1D algorithm, columns outside the
// target columns pushed into their reservoir rows). What remains is
// sequential by definition: the unsolved columns are filled one after the
// other, left to right, each from every token of the grid at once, and each
// fill changes the tokens the next one sees. One block per grid runs that
// loop with the grid's reservoir rows resident in shared memory, one half of
// its threads on each side of the band.
//
// The generalised 1D instance of receiver column j (Sec. III.E): an atom in a
// reservoir row v of a column at distance d sits on vertex v - d of column j
// above the band and on v + d below it, so that its Manhattan distance to any
// band trap of j is its distance along j. Tokens on one diagonal share a
// vertex. The vertices nearest the band are visited outward, layer by layer
// (layer k = vertex r0 - 1 - k above, r1 + k below; inside a layer the nearer
// column first, left before right): the first tokens met are the nearest,
// which is the order in which the optimal window takes them. The window
// itself is red-rec's split: a tokens from above, all band atoms of j, the
// rest from below, a of least total distance (largest a on ties), found by
// the discrete derivative of the convex cost.
//
// What bounds it: the chain from one receiver to the next, about seven
// barriers and as many shared-memory round trips. A side's nearest tokens are
// found without visiting cells one by one: a thread per column counts its
// tokens by layer (one shared add per token), a scan of the counts gives the
// cut-off layer and each layer's place in the list, a second pass puts the
// tokens into their layers, and within a layer (a column has at most one token
// in it) a token's rank is the number of smaller entries. The layers counted
// are the previous receiver's and a margin, more only when these do not
// suffice: the reservoirs change little from one receiver to the next. Sides
// of one warp (small grids, calls over very many) first walk the nearest cells
// in order, which costs fewer instructions while the reservoirs are full.
// Measured, against one warp per side walking cells, bisecting for the cut-off
// and sorting by a bitonic network: 427 x 256 1089 -> 208 us, 1024 x 1024 51.7
// -> 5.1 ms, 1024 grids of up to 256 x 256 4.1 -> 0.79 ms, 3000 of up to 64 x
// 64 324 -> 227 us.
#pragma once
#include "rr_internal.cuh"

namespace rrk {

// Token of a list: row in the upper 16 bits, column in the lower.
__device__ __forceinline__ int tok_row(int v) { return v >> 16; }
__device__ __forceinline__ int tok_col(int v) { return v & 0xffff; }

__device__ __forceinline__ int isqrt_floor(int g)
{
    int k = (int)sqrtf((float)g);
    while (k * k > g) --k;
    while ((k + 1) * (k + 1) <= g) ++k;
    return k;
}

// Walk order: cell g of one side is layer k = floor(sqrt(g)) (the vertex
// r0-1-k above the band, r1+k below it), index i = g - k*k in the layer:
// i = 0 is column j itself, i = 2d-1 column j-d, i = 2d column j+d, on row
// r0-1-k+d above the band or r1+k-d below it. Ascending g is the order in
// which the optimal window takes tokens (nearest vertex first, then the
// nearer column, left before right).
__device__ __forceinline__ void walk_cell(int g, int j, int r0, int r1, bool top, int *row, int *col)
{
    const int k = isqrt_floor(g);
    const int i = g - k * k;
    const int d = (i + 1) >> 1;
    *col = d == 0 ? j : ((i & 1) ? j - d : j + d);
    *row = top ? r0 - 1 - k + d : r1 + k - d;
}

// The nearest tokens of one side by visiting cells in order (one warp, 32
// cells at a time, maxIter times at most): the tokens held if `need` were
// found or no cell is left, else -1.
__device__ __forceinline__ int bird_walk(const uint32_t *bits, int Wp, int m, int n, int r0, int r1, int j, bool top, int need,
                                         int kmax, int maxIter, int lane, int32_t *list)
{
    const int gEnd = (kmax + 1) * (kmax + 1);
    int got = 0, g = 0;
    for (int it = 0; got < need && g < gEnd; ++it, g += 32) {
        if (it == maxIter) return -1;
        const int gl = g + lane;
        int row, col;
        walk_cell(gl, j, r0, r1, top, &row, &col);
        bool occ = false;
        if (gl < gEnd && col >= 0 && col < n && row >= 0 && row < m && (top ? row < r0 : row >= r1))
            occ = (bits[col * Wp + (row >> 5)] >> (row & 31)) & 1u;
        const unsigned bal = __ballot_sync(FULL, occ);
        const int rank = got + __popc(bal & ((1u << lane) - 1u));
        if (occ && rank < need) list[rank] = (row << 16) | col;
        got = min(need, got + __popc(bal));
    }
    return got;
}

// Position of a token of receiver j in the order in which the optimal window
// takes them, on one side of the band: layer k in the upper bits, then its
// place i in the layer: i = 0 is column j itself, i = 2d-1 column j-d, i = 2d
// column j+d, on row r0-1-k+d above the band or r1+k-d below it.
constexpr int KEY_I = 11;
static_assert(2 * RR_MAX_SIDE <= 1 << KEY_I, "places of a layer");
__device__ __forceinline__ uint32_t bird_key(int k, int c, int j)
{
    return (uint32_t)k << KEY_I | (uint32_t)(c < j ? 2 * (j - c) - 1 : 2 * (c - j));
}

// Barrier of one side's threads. (Immediate ids: a barrier number in a
// register claims all sixteen, and fewer blocks fit on an SM.)
__device__ __forceinline__ void side_sync(bool top, int T)
{
    if (T == 32) __syncwarp();
    else if (top) asm volatile("bar.sync 1, %0;" ::"r"(T) : "memory");
    else asm volatile("bar.sync 2, %0;" ::"r"(T) : "memory");
}

// One side of the band of one receiver: its threads (T of them, st the
// thread's number) call f(layer, column) for every token in the layers above
// `from` and up to `to`. While these reach over few columns, 2, 4 or 8 threads
// share one, each with some of every word's bits. A word's lowest and highest
// bit are taken together: the two searches' latencies overlap.
template <class F>
__device__ __forceinline__ void bird_tokens(const uint32_t *bits, int Wp, int m, int n, int r0, int r1, int j, bool top,
                                            int from, int to, int st, int T, F f)
{
    const int first = max(0, j - to), cols = min(n - 1, j + to) - first + 1;
    const int sh = cols > T / 2 ? 0 : cols > T / 4 ? 1 : cols > T / 8 ? 2 : 3;
    const uint32_t part = sh == 0 ? FULL : (1u << (32 >> sh)) - 1u << (st & ((1 << sh) - 1)) * (32 >> sh);
    for (int q = st >> sh; q < cols; q += T >> sh) {
        const int c = first + q, d = iabs(c - j);
        const int lo = top ? max(0, r0 - 1 - to + d) : max(r1, r1 + from + 1 - d);
        const int end = top ? min(r0, r0 - 1 - from + d) : min(m, r1 + to - d + 1);
        for (int w = lo >> 5; 32 * w < end; ++w) {
            // the layer of bit b: k0 - b above the band, k0 + b below it
            const int k0 = (top ? r0 - 1 - 32 * w : 32 * w - r1) + d;
            for (uint32_t x = bits[c * Wp + w] & part & row_mask(w, lo, end); x;) {
                const int b0 = __ffs(x) - 1, b1 = 31 - __clz(x);
                x = x & (x - 1u) & ~(1u << b1);
                f(top ? k0 - b0 : k0 + b0, c);
                if (b1 != b0) f(top ? k0 - b1 : k0 + b1, c);
            }
        }
    }
}

// The `need` nearest tokens of receiver j on one side, in the window's order,
// or all of them if fewer: into list; returns their number. hist: zero for
// every layer on entry; the layers up to *used are not on return. guess: the
// layers to count at first (on return: for the next receiver, the cut-off and
// as many more as it has grown by since the last one; a layer near it may hold
// as many tokens as the receiver needs). s_out: two words.
__device__ __forceinline__ int bird_side(const uint32_t *bits, int Wp, int m, int n, int r0, int r1, int j, bool top,
                                         int need, int32_t *list, uint32_t *keys, unsigned *hist, int *s_out, int st,
                                         int T, int *guess, int *last, int *used, bool *sparse)
{
    *used = -1;
    if (top ? r0 == 0 : r1 == m) return 0;
    const int lane = st & 31;
    const int kmax = (top ? r0 - 1 : m - 1 - r1) + max(j, n - 1 - j);     // no cell beyond this layer
    if (T == 32 && !*sparse) {
        const int got = bird_walk(bits, Wp, m, n, r0, r1, j, top, need, kmax, 8 + need / 8, lane, list);
        if (got >= 0) return got;
    }
    int from = -1, to = min(*guess, kmax), more = 2, K, total;
    for (;;) {
        bird_tokens(bits, Wp, m, n, r0, r1, j, top, from, to, st, T, [&](int k, int) { atomicAdd(&hist[k], 1u); });
        side_sync(top, T);
        if (st < 32) {
            // the first layer with `need` tokens up to it; the layers' places
            const int per = (to + 32) >> 5 | 1, k0 = lane * per, k1 = min(k0 + per, to + 1);
            int sum = 0;
#pragma unroll 4
            for (int k = k0; k < k1; ++k) sum += (int)hist[k];
            const int incl = warp_incl_scan(sum);
            const unsigned full = __ballot_sync(FULL, incl >= need);
            if (full || to == kmax) {
                int at = incl - sum, cut = 0x7fffffff, tot = 0;
#pragma unroll 4
                for (int k = k0; k < k1; ++k) {
                    const int c = (int)hist[k];
                    hist[k] = (unsigned)at;
                    at += c;
                    if (at >= need && cut == 0x7fffffff) { cut = k; tot = at; }
                }
                const int src = full ? __ffs(full) - 1 : 31;
                cut = __shfl_sync(FULL, full ? cut : kmax, src);
                tot = __shfl_sync(FULL, full ? tot : incl, src);
                if (lane == 0) { s_out[0] = cut; s_out[1] = tot; }
            } else if (lane == 0) {
                s_out[0] = -1;
            }
        }
        side_sync(top, T);
        K = s_out[0];
        total = s_out[1];
        if (K >= 0) break;
        from = to;
        to = min(kmax, to + more);
        more *= 2;
    }
    // tokens into their layers; a layer's entry ends at the next one's start
    bird_tokens(bits, Wp, m, n, r0, r1, j, top, -1, K, st, T,
                [&](int k, int c) { keys[atomicAdd(&hist[k], 1u)] = bird_key(k, c, j); });
    if (st < 3) keys[total + st] = FULL;
    side_sync(top, T);
    for (int t = st; t < total; t += T) {
        // (four entries at a time: those before the layer are all smaller,
        // those after it greater)
        const uint32_t x = keys[t];
        const int k = (int)(x >> KEY_I), b0 = (k > 0 ? (int)hist[k - 1] : 0) & ~3, b1 = (int)hist[k];
        int at = b0;
#pragma unroll 2
        for (int u = b0; u < b1; u += 4) {
            const uint4 y = *(const uint4 *)(keys + u);
            at += (y.x < x) + (y.y < x) + (y.z < x) + (y.w < x);
        }
        const int i = (int)(x & ((1u << KEY_I) - 1u)), d = (i + 1) >> 1;
        if (at < need) list[at] = (top ? r0 - 1 - k + d : r1 + k - d) << 16 | ((i & 1) ? j - d : j + d);
    }
    *guess = K + max(1, K - *last);
    *last = K;
    *sparse = (K + 1) * (K + 1) > 32 * (8 + need / 8);
    *used = to;
    return min(total, need);
}

// Every thread of the block calls it: T on each side of the band.
__device__ inline void s_bird(const Blk B, rr_instance *inst, JobWS *wsv, int count, int max_side)
{
    extern __shared__ __align__(16) uint32_t birdsm[];
    __shared__ int s_got[2], s_base, s_bad, s_nrecv, s_out[4];
    const int q = B.x;
    if (q >= count) return;
    rr_instance *I = &inst[q];
    if (!live(I)) return;
    JobWS &ws = wsv[q];
    const int m = I->m, n = I->n, W = (m + 31) >> 5;
    const int r0 = I->rect.r0, r1 = I->rect.r1, c0 = I->rect.c0, c1 = I->rect.c1, h = r1 - r0;
    const int threads = blockDim.x, T = threads >> 1;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, side = tid >= T ? 1 : 0;
    const BirdLayout Y(max_side);
    const int Wp = W | 1;                                                  // odd: neighbouring columns in different banks
    uint32_t *bits = birdsm;                                               // n * Wp words
    int32_t *topTok = (int32_t *)(birdsm + Y.lists), *botTok = topTok + max_side;
    uint32_t *keys = birdsm + Y.keys + side * Y.room;
    unsigned *hist = birdsm + Y.hist + side * 2 * max_side;
    // receivers in column order (column, band atoms, atoms above the band),
    // and the current receiver's band holes and band atom rows
    int16_t *recvCol = (int16_t *)(birdsm + Y.recv);
    int16_t *recvM = recvCol + max_side, *recvTop = recvM + max_side;
    int16_t *sHr = recvTop + max_side, *sOwn = sHr + max_side;

    // Feasibility (total surplus, Sec. III.C) and the offsets of the column
    // units, in column order.
    if (wid == 0) {
        int tot = 0, carry = 0;
        for (int base = 0; base < n; base += 32) {
            const int c = base + lane;
            int v = 0;
            if (c < n) { v = ws.col[c].nmoves; tot += ws.col[c].sigma; }
            const int incl = warp_incl_scan(v);
            if (c < n) ws.unitOff[c] = carry + incl - v;
            carry += __shfl_sync(FULL, incl, 31);
        }
        tot = warp_sum(tot);
        if (lane == 0) {
            ws.unitOff[n] = carry;
            s_base = carry;
            s_bad = tot < 0;
        }
    } else if (wid == 1) {
        int nr = 0;
        for (int base = c0; base < c1; base += 32) {
            const int c = base + lane;
            bool rc = false;
            int M = 0, T = 0;
            if (c < c1) { const ColInfo ci = ws.col[c]; rc = ci.kind == KIND_RECEIVER; M = ci.nband; T = ci.ntop; }
            const unsigned bal = __ballot_sync(FULL, rc);
            if (rc) {
                const int at = nr + __popc(bal & ((1u << lane) - 1u));
                recvCol[at] = (int16_t)c; recvM[at] = (int16_t)M; recvTop[at] = (int16_t)T;
            }
            nr += __popc(bal);
        }
        if (lane == 0) s_nrecv = nr;
    }
    // Reservoir rows after the column phase: solved target columns keep the
    // atoms outside their window, outer columns with enough atoms fill every
    // reservoir trap, the others are untouched. Band rows are never read.
    for (int i = tid; i < 4 * max_side; i += threads) birdsm[Y.hist + i] = 0u;
    for (int idx = tid; idx < n * W; idx += threads) {
        const int c = idx / W, w = idx - c * W;
        const ColInfo ci = ws.col[c];
        const uint32_t res = row_mask(w, 0, r0) | row_mask(w, r1, m);
        uint32_t x = ws.colbits[idx];
        if (ci.kind == KIND_OUTER_FULL) {
            x = res;
        } else if (ci.kind == KIND_TARGET_SOLVED) {
            const int16_t *rows = ws.atomRows + (size_t)c * m;
            const int topLim = ci.ptop > 0 ? rows[ci.ptop - 1] + 1 : 0;   // pool above: rows < topLim
            const int botLim = ci.pbot > 0 ? rows[ci.bbase] : m;           // pool below: rows >= botLim
            x &= row_mask(w, 0, topLim) | row_mask(w, botLim, m);
        }
        bits[c * Wp + w] = x & res;
    }
    __syncthreads();
    if (s_bad) {
        if (tid == 0) { I->status = RR_INFEASIBLE; I->n_moves = 0; }
        return;
    }

    const long long colTotal = s_base;
    const int nrecv = s_nrecv;
    long long done = 0;          // moves of the receiver units so far
    long long steps = 0;
    int guess = -1, last = 0;    // this side's layers to count, its last cut-off
    bool sparse = false;
    for (int u = 0; u < nrecv; ++u) {
        const int j = recvCol[u], M = recvM[u], ownTop = recvTop[u];
        const int need = h - M, nh = h - M;
        // this receiver's band holes and band atoms (read by the split and
        // the emission once the tokens are found): the first ones' loads are
        // in flight meanwhile
        const int16_t *ghr = ws.holeRows + (size_t)(j - c0) * h;
        const int16_t *gown = ws.atomRows + (size_t)j * m + ownTop;
        const int16_t hr0 = tid < nh ? ghr[tid] : (int16_t)0, own0 = tid < M ? gown[tid] : (int16_t)0;
        if (guess < 0) guess = last = 2 + (int)sqrtf(2.f * (float)need);
        int used;
        const int got = bird_side(bits, Wp, m, n, r0, r1, j, side == 0, need, side == 0 ? topTok : botTok, keys, hist,
                                  s_out + 2 * side, tid - side * T, T, &guess, &last, &used, &sparse);
        if (tid == side * T) s_got[side] = got;
        if (tid < nh) sHr[tid] = hr0;
        if (tid < M) sOwn[tid] = own0;
        for (int t = tid + threads; t < nh; t += threads) sHr[t] = ghr[t];
        for (int t = tid + threads; t < M; t += threads) sOwn[t] = gown[t];
        const int16_t *hr = sHr;
        __syncthreads();
        for (int k = tid - side * T; k <= used; k += T) hist[k] = 0u;
        // every warp finds the split: that is cheaper than another barrier
        const int nt = s_got[0], nb = s_got[1];
        int a = -1;
        if (nt + nb >= need) {
            const int lo = max(0, need - nb), hi = min(need, nt);
            // d cost / da: one more token from above (the a-th nearest)
            // and one fewer from below (the (need-a+1)-th nearest)
            a = split_search(lo, hi, [&](int aa) {
                const int tv = topTok[aa - 1], bv = botTok[need - aa];
                const int tpos = tok_row(tv) - iabs(tok_col(tv) - j);
                const int bpos = tok_row(bv) + iabs(tok_col(bv) - j);
                return (r0 + aa - 1 - tpos) + (2 * band_P(hr, nh, M, r0, r0 + aa - 1) - M) +
                       (r0 + h - need + aa - 1 - bpos);
            });
        }
        if (a < 0) {             // cannot happen when the total surplus is >= 0
            if (tid == 0) set_status(I, RR_ERR_INTERNAL);
            return;
        }
        // Targets r0 + k: k < a from above (nearest deepest), then the band
        // atoms in order, then from below (nearest shallowest). Emission as
        // every unit: toward larger rows deepest first, then toward smaller
        // rows shallowest first; isolated band atoms are dropped.
        const int kd_end = a + band_P(hr, nh, M, r0, r0 + a - 1);
        const int ku_start = a + band_P(hr, nh, M, r0, r0 + a);
        const long long base = colTotal + done;
        for (int k = tid; k < h; k += threads) {
            int row, col;
            if (k < a) { const int v = topTok[a - 1 - k]; row = tok_row(v); col = tok_col(v); }
            else if (k < a + M) { row = sOwn[k - a]; col = j; }
            else { const int v = botTok[k - a - M]; row = tok_row(v); col = tok_col(v); }
            int pos;
            if (k < kd_end) pos = kd_end - 1 - k;
            else if (k >= ku_start) pos = kd_end + (k - ku_start);
            else continue;
            const long long o = base + pos;
            if (o < I->cap_moves) store_move(&I->moves[o], row, col, r0 + k, j);
            steps += iabs(r0 + k - row) + iabs(j - col);
        }
        // the chosen tokens leave the reservoirs
        for (int l = tid; l < need; l += threads) {
            const int v = l < a ? topTok[l] : botTok[l - a];
            const int row = tok_row(v), col = tok_col(v);
            atomicAnd(&bits[col * Wp + (row >> 5)], ~(1u << (row & 31)));
        }
        done += kd_end + (h - ku_start);
        __syncthreads();
    }
    add_steps(I, steps);
    if (tid == 0) {
        const long long total = colTotal + done;
        I->n_moves = total;
        if (total > I->cap_moves) set_status(I, RR_ERR_CAPACITY);
    }
}

} // namespace rrk
