"""Workloads that the library's speed is measured on: what its users call, at the sizes they call it with.

Points are integer-valued float32 pairs in [0, 2^24), drawn on the GPU with
the distributions of synth/workloads.py: uniform in the square, an isotropic
normal (most points are discarded by the filter), a ring of width 64 and a
circumference with 2% distortion (the filter's worst cases).  Every case goes
through the package's public entry points.  A case's fields:

  op       hull     one hull of device points (`hull`)
           host     one hull of pinned host points (`ch_hull_host`)
           small    one hull without library allocations (`ch_hull_noalloc`)
           batched  many hulls packed back to back (`ch_hull_batched`)
           filter   the octagon filter alone, labels of all points (`filter_labels`)
           filter16 the same with the 16-direction polygon (`filter16_labels`)
           serve    a burst of requests through the server (`ch_submit` / `ch_poll`)
  kind     the distribution ("mix": each set or request draws its own)
  n        points (batched, serve: points of the largest set; sizes log-uniform in [lo, n])
  k        sets or requests
  shift    1: the points start 8 bytes past a 16-byte boundary, as a slice of a larger tensor does
  wait     hull: True reads the hull's size back (the default of `hull`), False leaves the result on the device
"""
import atexit
import math
import random

import numpy as np
import torch

import paper_2209_12310_gb300 as ch

LIMIT = 1 << 24
CENTER = float(1 << 23)
KINDS = ("uniform", "normal", "ring", "distorted")
STEP = 1 << 24                # points drawn at a time
SERVER_BYTES = 4 << 30        # the server's memory budget
EXACT_MOST = 3_000_000        # points of the largest case whose hull is computed on the host


def listed():
    return [
        # the smallest served request: launches and latency
        {"name": "hull_uniform_1k", "op": "hull", "kind": "uniform", "n": 1_000, "k": 1, "shift": 0, "wait": True},
        # a small hull inside a pipeline that stays on the device; ragged size
        {"name": "hull_normal_65k", "op": "hull", "kind": "normal", "n": 65_537, "k": 1, "shift": 0, "wait": False},
        # the ordinary single hull (fits in L2)
        {"name": "hull_uniform_1m", "op": "hull", "kind": "uniform", "n": 1_000_000, "k": 1, "shift": 0, "wait": True},
        # the filter's worst case at an ordinary size, a misaligned slice
        {"name": "hull_ring_1m", "op": "hull", "kind": "ring", "n": 1_000_003, "k": 1, "shift": 1, "wait": True},
        # the distorted circumference at the size the paper quotes it for
        {"name": "hull_distorted_10m", "op": "hull", "kind": "distorted", "n": 10_000_000, "k": 1, "shift": 0,
         "wait": True},
        # the headline workload: one large hull, nearly every point discarded
        {"name": "hull_normal_100m", "op": "hull", "kind": "normal", "n": 100_000_000, "k": 1, "shift": 0,
         "wait": True},
        # the largest worst case
        {"name": "hull_ring_100m", "op": "hull", "kind": "ring", "n": 100_000_000, "k": 1, "shift": 0, "wait": True},
        # a batch of the size a server forms under load
        {"name": "batched_40", "op": "batched", "kind": "mix", "n": 1_000_000, "lo": 1_000, "k": 40, "shift": 0},
        # the large batch of uneven sets
        {"name": "batched_4096", "op": "batched", "kind": "mix", "n": 1_000_000, "lo": 100, "k": 4096, "shift": 0},
        # the filter alone, labels and queue counts of every point
        {"name": "filter_normal_100m", "op": "filter", "kind": "normal", "n": 100_000_000, "k": 1, "shift": 0},
        # its 16-direction form, odd size and misaligned
        {"name": "filter16_uniform_10m", "op": "filter16", "kind": "uniform", "n": 10_000_019, "k": 1, "shift": 1},
        # a burst of requests from pinned host memory, polled until all are answered
        {"name": "serve_burst_32", "op": "serve", "kind": "mix", "n": 1_000_000, "lo": 1_000, "k": 32, "shift": 0},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choices(("hull", "batched", "filter", "filter16", "host", "small", "serve"),
                     weights=(10, 4, 2, 1, 2, 1, 1))[0]
    shift = int(rng.random() < 0.4)
    kind = rng.choice(KINDS)
    if op == "small":
        return {"op": op, "kind": kind, "n": _log_int(rng, 100, 8_000), "k": 1, "shift": shift}
    if op == "host":
        return {"op": op, "kind": kind, "n": _log_int(rng, 1_000, 10_000_000), "k": 1, "shift": 0}
    if op == "batched":
        lo = rng.choice((100, 1_000))
        k = _log_int(rng, 8, 2_048)
        return {"op": op, "kind": rng.choice(KINDS + ("mix", "mix")), "n": _log_int(rng, 10 * lo, 1_000_000),
                "lo": lo, "k": k, "shift": shift}
    if op == "serve":
        return {"op": op, "kind": "mix", "n": _log_int(rng, 100_000, 2_000_000), "lo": 1_000,
                "k": rng.randint(8, 48), "shift": 0}
    n = _log_int(rng, 1_000, 100_000_000)
    case = {"op": op, "kind": kind, "n": n, "k": 1, "shift": shift}
    if op == "hull":
        case["wait"] = rng.random() < 0.5
    return case


# ---------------------------------------------------------------------------
# Inputs

def _fill(out, kind, gen):
    """Draws out (m, 2) float32 on the GPU."""
    for s in range(0, out.shape[0], STEP):
        part = out[s:s + STEP]
        m = part.shape[0]
        if kind == "uniform":
            part.copy_(torch.randint(0, LIMIT, (m, 2), generator=gen, device="cuda", dtype=torch.int32))
        elif kind == "normal":
            p = torch.randn((m, 2), generator=gen, device="cuda", dtype=torch.float64)
            part.copy_(p.mul_(float(1 << 21)).add_(CENTER).round_().clamp_(0.0, LIMIT - 1.0))
        else:
            a = torch.rand(m, generator=gen, device="cuda", dtype=torch.float64).mul_(2.0 * math.pi)
            r = torch.rand(m, generator=gen, device="cuda", dtype=torch.float64)
            r = CENTER - 64.0 * r if kind == "ring" else CENTER * (1.0 - 0.02 * r)
            part[:, 0].copy_(torch.cos(a).mul_(r).add_(CENTER).round_().clamp_(0.0, LIMIT - 1.0))
            part[:, 1].copy_(torch.sin(a).mul_(r).add_(CENTER).round_().clamp_(0.0, LIMIT - 1.0))


def _generator(seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    return gen


def _empty_points(n, shift):
    return torch.empty((n + shift, 2), dtype=torch.float32, device="cuda")[shift:]


def _sets(case):
    """Sizes and distributions of a case's sets, and their offsets: they belong
    to the case, the points to the seed."""
    plan = random.Random("%d %d %d %s" % (case["k"], case["n"], case["lo"], case["kind"]))
    sizes, kinds = [], []
    for _ in range(case["k"]):
        sizes.append(_log_int(plan, case["lo"], case["n"]))
        kinds.append(plan.choice(KINDS[:3]) if case["kind"] == "mix" else case["kind"])
    offsets = np.zeros(case["k"] + 1, dtype=np.int64)
    offsets[1:] = np.cumsum(sizes)
    return sizes, kinds, offsets


def _packed(case, seed):
    sizes, kinds, offsets = _sets(case)
    gen = _generator(seed)
    pts = _empty_points(int(offsets[-1]), case["shift"])
    for kind in KINDS:   # one draw per distribution, then the sets' shares
        mine = [i for i in range(case["k"]) if kinds[i] == kind]
        if not mine:
            continue
        src = torch.empty((sum(sizes[i] for i in mine), 2), dtype=torch.float32, device="cuda")
        _fill(src, kind, gen)
        for i, part in zip(mine, src.split([sizes[i] for i in mine])):
            pts[offsets[i]:offsets[i + 1]] = part
    return pts, offsets


def _points(case, seed):
    pts = _empty_points(case["n"], case["shift"])
    _fill(pts, case["kind"], _generator(seed))
    return pts


_servers = {}


def _server():
    """One server for the process, as a serving program keeps it."""
    if "srv" not in _servers:
        _servers["srv"] = ch.ch_server_create(SERVER_BYTES, torch.cuda.current_device())
        atexit.register(lambda: ch.ch_server_destroy(_servers.pop("srv")))
    return _servers["srv"]


def prepare(case, seed):
    op = case["op"]
    state = {"op": op}
    if op in ("batched", "serve"):
        pts, offsets = _packed(case, seed)
        total = int(offsets[-1])
        if op == "batched":
            state.update(pts=pts, offsets=torch.from_numpy(offsets).cuda(), host_offsets=torch.from_numpy(offsets),
                         k=case["k"], out_idx=torch.full((total,), -1, dtype=torch.int32, device="cuda"),
                         out_n=torch.zeros(case["k"], dtype=torch.int64, device="cuda"))
        else:
            state.update(srv=_server(), pts=pts.cpu().pin_memory(), offsets=offsets.tolist(),
                         out_idx=torch.full((total,), -1, dtype=torch.int32))
        return state
    pts = _points(case, seed)
    if op == "host":
        state.update(pts=pts.cpu().pin_memory(), out_idx=torch.full((case["n"],), -1, dtype=torch.int32).pin_memory(),
                     out_n=torch.zeros(1, dtype=torch.int64))
        return state
    state["pts"] = pts
    if op in ("hull", "small"):   # results go to the program's own buffers
        state.update(out_idx=torch.full((case["n"],), -1, dtype=torch.int32, device="cuda"),
                     out_n=torch.zeros(1, dtype=torch.int64, device="cuda"))
    if op == "hull":
        state["wait"] = case["wait"]
    return state


# ---------------------------------------------------------------------------
# One pass

def run(state):
    op, pts = state["op"], state["pts"]
    if op == "hull":
        ch.hull(pts, out_idx=state["out_idx"], out_n=state["out_n"], sync=state["wait"])
        return state["out_idx"], state["out_n"]
    if op == "batched":
        ch.ch_hull_batched(pts.data_ptr(), state["offsets"].data_ptr(), state["k"], state["out_idx"].data_ptr(),
                           state["out_n"].data_ptr(), state["host_offsets"].data_ptr(),
                           torch.cuda.current_stream().cuda_stream)
        return state["out_idx"], state["out_n"]
    if op == "filter":
        return ch.filter_labels(pts)
    if op == "filter16":
        return ch.filter16_labels(pts)
    if op == "small":
        ch.load().ch_hull_noalloc(pts.data_ptr(), pts.shape[0], state["out_idx"].data_ptr(),
                                  state["out_n"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        return state["out_idx"], state["out_n"]
    if op == "host":
        ch.ch_hull_host(pts.data_ptr(), pts.shape[0], state["out_idx"].data_ptr(), state["out_n"].data_ptr(),
                        torch.cuda.current_stream().cuda_stream)
        return state["out_idx"], state["out_n"]
    # serve: submit the burst, poll until every request is answered
    srv, offsets, out = state["srv"], state["offsets"], state["out_idx"]
    base, dst = pts.data_ptr(), out.data_ptr()
    waiting = []
    for i in range(len(offsets) - 1):
        o, n = offsets[i], offsets[i + 1] - offsets[i]
        status, ticket = ch.ch_submit(srv, base + 8 * o, n)
        if status != ch.CH_OK:
            raise ch.CHError(status, "ch_submit")
        waiting.append((i, ticket))
    sizes = [0] * len(waiting)
    while waiting:
        still = []
        for i, ticket in waiting:
            o = offsets[i]
            status, h = ch.ch_poll(srv, ticket, dst + 4 * o, offsets[i + 1] - o)
            if status == ch.CH_PENDING:
                still.append((i, ticket))
            elif status != ch.CH_OK:
                raise ch.CHError(status, "ch_poll")
            else:
                sizes[i] = h
        waiting = still
    return out, np.array(sizes, dtype=np.int64)


def work(case):
    """Every point read once (8 bytes); the labels written once (1 byte).  The
    hulls' own bytes are not counted: a few KB beside the points."""
    if case["op"] in ("batched", "serve"):
        total = int(_sets(case)[2][-1])
        return {"bytes": 8 * total + 16 * case["k"], "flops": 0}
    per = 9 if case["op"] in ("filter", "filter16") else 8
    return {"bytes": per * case["n"], "flops": 0}


# ---------------------------------------------------------------------------
# The same by plain numpy in 64 bits

def _hull64(pts):
    """Indices of the strictly convex vertices, counter-clockwise from the
    lexicographically smallest; the lowest index of repeated coordinates."""
    p = pts.astype(np.int64)
    # candidates: points not strictly inside the polygon of 64 directional extremes
    ang = np.arange(64) * (2.0 * math.pi / 64)
    ext = [int(np.argmax(p[:, 0] * c + p[:, 1] * s)) for c, s in zip(np.cos(ang), np.sin(ang))]
    keep = np.ones(len(p), dtype=bool)
    corners = [p[e] for j, e in enumerate(ext) if not np.array_equal(p[e], p[ext[j - 1]])]
    if len(corners) >= 3:
        inside = np.ones(len(p), dtype=bool)
        for a, b in zip(corners, corners[1:] + corners[:1]):
            inside &= (b[0] - a[0]) * (p[:, 1] - a[1]) - (b[1] - a[1]) * (p[:, 0] - a[0]) > 0
        keep = ~inside
    cand = np.nonzero(keep)[0]
    cand = cand[np.lexsort((cand, p[cand, 1], p[cand, 0]))]
    xy = p[cand]
    first = np.ones(len(cand), dtype=bool)
    first[1:] = np.any(xy[1:] != xy[:-1], axis=1)
    cand, xy = cand[first].tolist(), xy[first].tolist()
    if len(cand) <= 2:
        return np.array(cand, dtype=np.int64)

    def chain(order):
        got = []
        for j in order:
            x, y = xy[j]
            while len(got) >= 2:
                (ax, ay), (bx, by) = xy[got[-2]], xy[got[-1]]
                if (bx - ax) * (y - ay) - (by - ay) * (x - ax) > 0:
                    break
                got.pop()
            got.append(j)
        return got

    lower, upper = chain(range(len(cand))), chain(range(len(cand) - 1, -1, -1))
    return np.array([cand[j] for j in lower[:-1] + upper[:-1]], dtype=np.int64)


def exact(case, seed):
    op = case["op"]
    if op in ("filter", "filter16"):
        return None   # whole numbers only, no arithmetic to be off by
    total = int(_sets(case)[2][-1]) if op in ("batched", "serve") else case["n"]
    if total > EXACT_MOST:
        return None
    if op in ("batched", "serve"):
        pts, offsets = _packed(case, seed)
        pts = pts.cpu().numpy()
        hulls = [_hull64(pts[offsets[i]:offsets[i + 1]]) for i in range(case["k"])]
        out = np.full(total, -1, dtype=np.int64)
        for o, h in zip(offsets, hulls):
            out[o:o + len(h)] = h
        return out, np.array([len(h) for h in hulls], dtype=np.int64)
    h = _hull64(_points(case, seed).cpu().numpy())
    out = np.full(total, -1, dtype=np.int64)
    out[:len(h)] = h
    return out, np.array([len(h)], dtype=np.int64)
