"""What the framework is measured on: the calls its users make, through its
public entry points, over the range of sizes, planners, layouts and modes
that those calls accept.

A case is one kind of call (`entry`) on seeded random grids:

  one      rr_plan_one: one grid planned and batched by one kernel launch
  noalloc  rr_plan_noalloc: one grid planned without a context
  plan     rr_plan_mode, with `batch` followed by rr_batch
  batched  rr_plan_batched over `count` grids (plans only, or with `batch`
           plans and batches; `graph`: replayed from a captured graph)
  served   rr_serve_*: `count` requests submitted at once, every result read

Grids are loaded at random with fill `p` (batched: per grid uniform in
[p, p_hi]); `geometry` gives the target: "centred" (the centred rectangle of
`target` times each side), "paper" (n columns, ceil(n / 0.6) rows, full-width
target of n rows) or "chain" (m x 1, centred target of m / 2).

Every output is whole numbers: moves, batches, members, counts and statuses.
"""
import math
import os

import numpy as np
import torch

# Servers keep a dozen streams busy: as many hardware queues as streams, as
# the server's documentation asks for (read when the context is created).
os.environ.setdefault("CUDA_DEVICE_MAX_CONNECTIONS", "32")

import paper_2504_06182_gb300 as rr
from paper_2504_06182_gb300.planner import Planner, device_view, pack_instances, unpack_instances


def listed():
    return [
        # one reconfiguration cycle of today's arrays: the smallest call, where latency counts
        case("one-32", "one", m=32, n=32, target=20 / 32, layout="u8"),
        # the same cycle on a larger, oblong array, bit-packed, planned with bird
        case("one-bird-97x120", "one", m=97, n=120, target=0.7, layout="bits32", bird=True),
        # a control loop that must not allocate: the paper's geometry at 32 target columns
        case("noalloc-paper-32", "noalloc", m=54, n=32, geometry="paper", p=0.62, layout="u8"),
        # planning alone at the paper's largest size, with the planner that wants the most work
        case("plan-bird-paper-256", "plan", m=427, n=256, geometry="paper", p=0.62, layout="bits32", bird=True),
        # one ordinary large array: plan, then batch
        case("plan-batch-256", "plan", m=256, n=256, target=180 / 256, layout="bits32", batch=True),
        # odd sizes, bytes, strict reservoirs
        case("plan-batch-strict-389x501", "plan", m=389, n=501, target=0.58, layout="u8", batch=True, strict=True),
        # the largest array the framework takes
        case("plan-batch-1024", "plan", m=1024, n=1024, target=720 / 1024, layout="bits32", batch=True),
        # thousands of arrays of mixed sizes per call: a simulation study's step
        case("batched-4096", "batched", count=4096, lo=32, hi=256, step=16, p=0.5, p_hi=0.7, layout="bits32",
             batch=True),
        # the same with bird on fewer arrays, replayed from a graph as a control loop does
        case("batched-bird-graph-1024", "batched", count=1024, lo=32, hi=256, step=16, p=0.5, p_hi=0.7,
             layout="bits32", batch=True, bird=True, graph=True),
        # plans without batches, odd sides, bytes: a study of success rates
        case("batched-plan-2000", "batched", count=2000, lo=33, hi=251, step=2, p=0.55, p_hi=0.65, layout="u8"),
        # many independent 1D chains
        case("chains-16384", "batched", count=16384, lo=1024, hi=1024, step=1, geometry="chain", layout="u8"),
        # a burst of requests from many users, host grids in, results out
        case("served-48", "served", count=48, lo=64, hi=512, step=16, layout="bits32", batch=True),
    ]


def case(name, entry, m=0, n=0, count=1, lo=0, hi=0, step=1, geometry="centred", target=0.7, p=0.6, p_hi=0.0,
         layout="u8", batch=False, bird=False, strict=False, graph=False):
    c = dict(entry=entry, m=m, n=n, count=count, lo=lo, hi=hi, step=step, geometry=geometry, target=target, p=p,
             p_hi=max(p, p_hi), layout=layout, batch=batch or entry == "one", bird=bird, strict=strict, graph=graph)
    return dict(c, name=name) if name else c


def draw(rng):
    def log_int(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    def sides(a, b):
        m = log_int(a, b)
        return m, max(a, min(b, int(round(m * rng.uniform(0.6, 1.6)))))

    entry = rng.choice(("one", "noalloc", "plan", "plan", "batched", "batched", "chains", "served"))
    layout = rng.choice(("u8", "bits32"))
    bird = rng.random() < 0.35
    strict = rng.random() < 0.25
    target = rng.uniform(0.5, 0.58) if strict else rng.uniform(0.5, 0.7)
    p = rng.uniform(0.58, 0.7)
    if entry in ("one", "noalloc"):
        m, n = sides(12, 256)
        return case("", entry, m=m, n=n, target=target, p=p, layout=layout, bird=bird and entry == "one",
                    strict=strict and entry == "one")
    if entry == "plan":
        if rng.random() < 0.3:
            n = log_int(24, 512)
            return case("", "plan", m=(5 * n + 2) // 3, n=n, geometry="paper", p=rng.uniform(0.62, 0.7), layout=layout, bird=bird,
                        batch=rng.random() < 0.4 and n <= 320)
        m, n = sides(24, 1024)
        return case("", "plan", m=m, n=n, target=target, p=p, layout=layout, bird=bird, strict=strict,
                    batch=max(m, n) <= 700 and rng.random() < 0.7)
    if entry == "chains":
        side = log_int(48, 1024)
        return case("", "batched", count=log_int(300, 16384), lo=side, hi=side, geometry="chain", layout=layout)
    hi = log_int(48, 256 if entry == "batched" else 512)
    lo = max(24, int(hi * rng.uniform(0.1, 0.9)))
    step = rng.choice((1, 2, 16))
    if entry == "served":
        return case("", "served", count=rng.randint(8, 48), lo=lo, hi=hi, step=step, p=p, layout=layout, batch=True)
    return case("", "batched", count=log_int(60, 3000), lo=lo, hi=hi, step=step, target=target, p=rng.uniform(0.5, 0.6),
                p_hi=rng.uniform(0.6, 0.7), layout=layout, bird=bird, strict=strict, batch=rng.random() < 0.75,
                graph=rng.random() < 0.3)


# ------------------------------------------------------------------ inputs

def rect_of(c, m, n):
    """Half-open target rectangle (r0, c0, r1, c1)."""
    if c["geometry"] == "paper":
        h, w = n, n
    elif c["geometry"] == "chain":
        h, w = m // 2, 1
    else:
        h, w = max(1, int(c["target"] * m)), max(1, int(c["target"] * n))
    r0, c0 = (m - h) // 2, (n - w) // 2
    return (r0, c0, r0 + h, c0 + w)


def pack_bits(u8):
    """(..., n) 0/1 bytes -> (..., ceil(n / 32)) int32 words, least significant bit first."""
    n = u8.shape[-1]
    w = (n + 31) // 32
    x = torch.nn.functional.pad(u8, (0, 32 * w - n)).reshape(*u8.shape[:-1], w, 32).to(torch.int64)
    x = (x << torch.arange(32, device=u8.device)).sum(-1)
    return torch.where(x >= 1 << 31, x - (1 << 32), x).to(torch.int32)


def random_grids(c, shapes, seed, device):
    """One contiguous grid of each (m, n) in `shapes`, in the case's layout."""
    gen = torch.Generator(device=device)
    gen.manual_seed(seed * 1000003 + 17)
    fill = torch.rand(len(shapes), generator=gen, device=device) * (c["p_hi"] - c["p"]) + c["p"]
    out = [None] * len(shapes)
    by_shape = {}
    for i, s in enumerate(shapes):
        by_shape.setdefault(s, []).append(i)
    for (m, n), ids in sorted(by_shape.items()):
        p = fill[torch.tensor(ids, device=device)].reshape(-1, 1, 1)
        g = (torch.rand((len(ids), m, n), generator=gen, device=device) < p).to(torch.uint8)
        g = pack_bits(g) if c["layout"] == "bits32" else g
        for k, i in enumerate(ids):
            out[i] = g[k]
    return out


def shapes_of(c):
    if c["entry"] not in ("batched", "served"):
        return [(c["m"], c["n"])]
    if c["geometry"] == "chain":
        return [(c["lo"], 1)] * c["count"]
    pick = np.random.RandomState(7).choice(np.arange(c["lo"], c["hi"] + 1, c["step"]), c["count"])
    return [(int(s), int(s)) for s in pick]


def steps_room(c, shapes):
    """Room for the batches of all grids: elementary steps, at most. About
    0.07 (red-rec) to 0.1 (bird) of traps times side are needed per feasible
    grid; of many thinly loaded grids about half are feasible."""
    rate = 0.16 if c["p"] >= 0.58 or len(shapes) < 500 else 0.07 if not c["bird"] else 0.1
    return int(rate * sum(m * n * max(m, n) for m, n in shapes)) + 4096


def flags_of(c):
    return ((rr.RR_BIRD if c["bird"] else 0) | (rr.RR_STRICT_RESERVOIR if c["strict"] else 0))


LAYOUT = {"u8": rr.RR_U8, "bits32": rr.RR_BITS32}


# --------------------------------------------------------------- the calls

class State:
    """What a program that makes these calls keeps: a planner or a server,
    its grids and its output buffers."""

    def __init__(self, c):
        self.case, self.layout, self.flags = c, LAYOUT[c["layout"]], flags_of(c)
        self.planner = self.server = None

    def __del__(self):
        if self.server:
            torch.cuda.synchronize()
            rr.rr_serve_close(self.server)
            self.server = None
        if self.planner:
            self.planner.close()


def prepare(c, seed):
    s = State(c)
    return {"served": prepare_served, "batched": prepare_batched}.get(c["entry"], prepare_single)(s, c, seed)


def zeros(rows, width):
    return torch.zeros((rows, width) if width > 1 else (rows,), dtype=torch.int32, device="cuda")


def prepare_single(s, c, seed):
    m, n = c["m"], c["n"]
    s.rect = rect_of(c, m, n)
    s.grid, = random_grids(c, [(m, n)], seed, "cuda")
    s.moves = zeros(2 * m * n, 4)
    if c["entry"] != "noalloc":
        s.planner = Planner(arena_bytes=(256 << 20) + 3200 * m * n if c["batch"] else 64 << 20)
    if c["batch"]:
        s.room = steps_room(c, [(m, n)])
        s.ops, s.members = zeros(s.room, 3), zeros(s.room, 1)
    return s


def run_single(s, c):
    m, n = c["m"], c["n"]
    if c["entry"] == "noalloc":
        return [*rr.rr_plan_noalloc(s.grid, s.layout, m, n, s.rect, s.moves, len(s.moves)), s.moves]
    if c["entry"] == "one":
        r = rr.rr_plan_one(s.planner.ctx, s.grid, s.layout, m, n, s.rect, s.flags | rr.RR_WITH_BATCH, s.moves,
                           len(s.moves), s.ops, s.room, s.members, s.room)
        return [*r, s.moves, s.ops, s.members]
    st, k = rr.rr_plan_mode(s.planner.ctx, s.grid, s.layout, m, n, s.rect, s.flags, s.moves, len(s.moves))
    if not c["batch"]:
        return [st, k, s.moves]
    r = rr.rr_batch(s.planner.ctx, s.moves, k, m, n, s.ops, s.room, s.members, s.room)
    return [st, k, *r, s.moves, s.ops, s.members]


def prepare_batched(s, c, seed):
    shapes = shapes_of(c)
    count = len(shapes)
    s.max_side = max(max(x) for x in shapes)
    s.grids = random_grids(c, shapes, seed, "cuda")
    cells = sum(m * n for m, n in shapes)
    side = s.max_side
    arena = (512 << 20) + 24 * cells + 2048 * 16 * count
    s.planner = Planner(arena_bytes=arena + (cells * (160 + 2 * side) if c["batch"] else 0))
    entries = [dict(grid=g, layout=s.layout, m=m, n=n, rect=rect_of(c, m, n)) for g, (m, n) in zip(s.grids, shapes)]

    def call(flags):
        s.inst = pack_instances(entries)
        st = rr.rr_plan_batched(s.planner.ctx, s.inst, count, s.max_side, flags)
        if st != rr.RR_OK:
            raise rr.RRError(st, rr.rr_last_error(s.planner.ctx))
        return unpack_instances(s.inst, count)

    def give(counts, **bufs):
        """Each grid's part of the buffers, packed grid after grid, to its entry."""
        at = np.concatenate([[0], np.cumsum(counts)])
        for key, b in bufs.items():
            if at[-1] >= len(b):
                raise RuntimeError("room for %d, %d needed" % (len(b), at[-1]))
            for i, e in enumerate(entries):
                e[key], e["cap_" + key] = b[int(at[i]):int(at[i]) + 1], int(counts[i])

    # a program sizes its buffers by planning: moves first, then elementary steps
    s.moves = zeros((2 if c["geometry"] != "chain" else 1) * cells + 1, 4)
    give([x.n_moves for x in call(s.flags)], moves=s.moves)
    s.ops = s.members = None
    if c["batch"]:
        total = steps_room(c, shapes)
        s.ops, s.members = zeros(total, 3), zeros(total, 1)
        give([x.n_steps for x in call(s.flags)], ops=s.ops, members=s.members)
    s.inst = pack_instances(entries)
    s.call_flags = s.flags | (rr.RR_WITH_BATCH if c["batch"] else 0) | (rr.RR_GRAPH if c["graph"] else 0)
    return s


def run_batched(s, c):
    st = rr.rr_plan_batched(s.planner.ctx, s.inst, c["count"], s.max_side, s.call_flags)
    counts = s.inst.view(torch.int64).reshape(c["count"], 16)[:, 11:16]   # moves, steps, batches, members, status
    return [st, counts, s.moves] + ([s.ops, s.members] if c["batch"] else [])


def prepare_served(s, c, seed):
    shapes = shapes_of(c)
    s.requests = [(np.ascontiguousarray(g.cpu().numpy()), m, n, rect_of(c, m, n))
                  for g, (m, n) in zip(random_grids(c, shapes, seed, "cuda"), shapes)]
    top = max(max(x) for x in shapes)
    s.server = rr.rr_serve_open(max_side=top, slots=64, streams=12, max_wave=8, flags=rr.RR_WITH_BATCH | s.flags,
                                arena_bytes=2 << 30, heap_bytes=8 << 30)
    room = steps_room(c, shapes)
    s.out = zeros(2 * sum(m * n for m, n in shapes), 4), zeros(room, 3), zeros(room, 1)
    return s


def run_served(s, c):
    tickets = [rr.rr_serve_submit(s.server, g, s.layout, m, n, rect)[1] for g, m, n, rect in s.requests]
    counts, at = [], [0, 0, 0]
    for t in tickets:
        st, r = rr.rr_serve_poll(s.server, t, timeout_us=60_000_000)
        if st != rr.RR_OK:
            raise rr.RRError(st, "rr_serve_poll")
        counts.append((r.status, r.n_moves, r.n_steps, r.n_ops, r.n_members))
        parts = (r.d_moves, (r.n_moves, 4)), (r.d_ops, (r.n_ops, 3)), (r.d_members, (r.n_members,))
        for i, (ptr, shape) in enumerate(parts):       # into the program's own buffers, request after request
            s.out[i][at[i]:at[i] + shape[0]].copy_(device_view(ptr, shape))
            at[i] += shape[0]
    torch.cuda.current_stream().synchronize()          # the results are copied: their memory goes back to the server
    for t in tickets:
        rr.rr_serve_release(s.server, t)
    return [np.array(counts), *s.out]


def run(s):
    return {"served": run_served, "batched": run_batched}.get(s.case["entry"], run_single)(s, s.case)


# ------------------------------------------------------------ work, exact

def work(c):
    """Each grid read once, each move (16 bytes), batch (12) and member (4)
    written once. How many there are depends on the loading; the rates per
    grid are fits to counts of sample grids (moves per trap, members and
    batches per trap and side)."""
    shapes = shapes_of(c)
    total = 0.0
    for m, n in shapes:
        cells = m * n
        grid = cells if c["layout"] == "u8" else 4 * m * ((n + 31) // 32)
        share = 0.5 if c["p"] < 0.58 else 1.0       # thinly loaded grids: about half are infeasible and get no moves
        moves = {"centred": 0.57, "paper": 0.56, "chain": 0.5}[c["geometry"]] * cells * share
        if c["strict"]:                             # smaller targets: few receivers, long lines of tokens
            share *= 0.35
        side = math.sqrt(cells)
        members = (0.1 if c["bird"] else 0.07) * cells * side * share
        ops = (0.012 if c["strict"] else 0.078 if c["bird"] else 0.043) * cells * side * share
        total += grid + 16 * moves + (12 * ops + 4 * members if c["batch"] else 0)
    # integer work only: no floating-point operations
    return {"bytes": total, "flops": 0}


def exact(c, seed):
    """Every output is a whole number and has to be equal: there is no
    rounding that a 64-bit calculation could show."""
    return None


if __name__ == "__main__":
    for x in listed():
        print(x["name"], "%.3g MB" % (work(x)["bytes"] / 1e6))
