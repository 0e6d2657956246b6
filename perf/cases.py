"""Performance cases of the embedding table: what a user's program has it do, at the sizes it does it.

Five kinds of pass, each through the package's public entry points (binding.py):

  pull   serving: mono_lookup_pool of a batch that nobody announced; the table only changes between requests
  train  the training loop that knows its batches ahead: push the gradients of the batch that was pulled last, sweep (one
         slice of a long-running table, the whole of a drifting one), announce and pull the next batch, and have the one
         after it grouped meanwhile
  push   training without announcements: MonoTable.apply_grads, then the rows of the batch's distinct IDs read back one
         by one (bags of one ID), as a job that ships trained rows to the serving side does
  group  many tables of uneven size and of mixed dims through the grouped calls, one table swept per step
  host   the training loop of a program whose batches live in pinned host memory (mono_*_host)

A state keeps a short ring of batches, so that successive passes see different IDs.  There are two kinds of tables:

  ttl >= 1000  a long-running table: the popular half of its rows' worth of IDs own rows, as many again are on probation
               (placed in random order), and nothing expires while the case runs.  The ring's IDs that were unknown
               enter on its first rounds.
  small ttl    a stream that drifts: the ring is longer than the ttl, so an ID that only one batch holds is inserted,
               perhaps admitted, expired and forgotten before it comes round again, for as long as the case runs.  `new` is
               the share of the ranks that carry an identity of their own in each batch.

IDs are Zipf ranks mixed into 64 bits, as in workload.py; gradients are N(0, 0.01^2).  All state is fp32.
"""
import math

import numpy as np
import torch

from paper_2209_07663_b200 import binding as mb
from paper_2209_07663_b200 import workload as wl

LONG_TTL = 1 << 20
UNIVERSE = 16            # distinct IDs of the stream, as a multiple of the table's rows
GROUP_DIMS = (8, 16, 32, 64)


def _case(name, kind, bags, lens, max_len, dim, rows, zipf, threshold, ttl=LONG_TTL, new=0.0, sketch=False, tables=1):
    return {"name": name, "kind": kind, "bags": bags, "lens": lens, "max_len": max_len, "dim": dim, "rows": rows,
            "zipf": zipf, "threshold": threshold, "ttl": ttl, "new": new, "sketch": sketch, "tables": tables}


def listed():
    return [
        # one ranking request: 8 candidates of 26 feature slots against a medium table; latency is all that counts
        _case("pull_request", "pull", 208, "uniform", 8, 32, 1 << 22, 1.05, 3),
        # a serving batch of the `medium` configuration's shape
        _case("pull_medium", "pull", 8192 * 26, "uniform", 8, 32, 1 << 22, 1.05, 3),
        # offline scoring with the `large` configuration's batch: 1.6 M bags, 8 M IDs, rows of 256 bytes
        _case("pull_large", "pull", 16384 * 100, "geometric", 20, 64, 1 << 24, 1.05, 5),
        # wide rows and long bags (user histories), a width that fills no power of two of lanes, an odd bag count
        _case("pull_wide", "pull", 40961, "uniform", 64, 200, 1 << 20, 1.1, 2),
        # the `tiny` configuration: an online trainer's small batches, where a step is launches
        _case("train_tiny", "train", 8192, "uniform", 4, 16, 1 << 17, 1.1, 2),
        # the `medium` configuration
        _case("train_medium", "train", 8192 * 26, "uniform", 8, 32, 1 << 22, 1.05, 3),
        # the `large` configuration's batch, on a table a quarter of its rows so that several fit the card at once
        _case("train_large", "train", 16384 * 100, "geometric", 20, 64, 1 << 24, 1.05, 5),
        # the `drift` configuration's batch: insertions, displacements, admissions and expiries in every step
        _case("train_drift", "train", 16384 * 50, "geometric", 20, 32, 1 << 19, 1.2, 3, ttl=4, new=0.3),
        # the probabilistic admission filter in place of exact counters, on the `medium` batch with drift
        _case("train_sketch", "train", 8192 * 26, "uniform", 8, 32, 1 << 21, 1.05, 3, ttl=4, new=0.1, sketch=True),
        # a batch that was not announced, odd in every size, on a table whose rows are not a power of two of lanes wide
        _case("push_odd", "push", 60013, "geometric", 20, 100, 1500007, 1.0, 3),
        # many small tables (two feature slots each) in one launch per step of the path
        _case("group_small", "group", 8192, "uniform", 4, 64, 1 << 17, 1.1, 2, tables=64),
        # the `medium` batch from and to pinned host memory
        _case("host_medium", "host", 8192 * 26, "uniform", 8, 32, 1 << 22, 1.05, 3),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("pull", "pull", "train", "train", "train", "push", "group", "host"))
    lens, max_len = rng.choice((("uniform", 4), ("uniform", 8), ("geometric", 20), ("uniform", rng.randint(1, 64))))
    mean = _mean_len({"lens": lens, "max_len": max_len})
    dim = 4 * log_int(2, 64)
    most = {"pull": 16384 * 100, "train": 16384 * 100, "push": 16384 * 25, "group": 8192, "host": 16384 * 25}[kind]
    # no dearer than the largest listed case: its IDs and its pooled values at most, half of them where the batch is read back
    ids, values = (8.1e6, 16384 * 100 * 64) if kind in ("pull", "train") else (4e6, 16384 * 25 * 64)
    tables = rng.randint(2, 64) if kind == "group" else 1
    # rows from three times the batch's IDs (the ring's unknown IDs must find free ones) to a table of 9 GB
    most_rows = min(1 << 17 if kind == "group" else 1 << 24, (9 << 30) // (8 * dim))
    bags = min(log_int(64, most), int(ids / mean / tables), int(values / dim / tables), int((most_rows - 4096) / 3 / mean))
    rows = log_int(3 * bags * mean + 4096, most_rows)
    drifts = kind == "train" and rng.random() < 0.3
    return {"kind": kind, "bags": bags, "lens": lens, "max_len": max_len, "dim": dim, "rows": rows,
            "zipf": round(rng.uniform(0.95, 1.3), 3), "threshold": rng.randint(1, 5), "ttl": 4 if drifts else LONG_TTL,
            "new": round(rng.uniform(0.0, 0.3), 3) if drifts else 0.0, "sketch": kind == "train" and rng.random() < 0.2,
            "tables": tables}


# ---- inputs -----------------------------------------------------------------

def _mean_len(c):
    return (1 + c["max_len"]) / 2 if c["lens"] == "uniform" else wl._mean_bag_len(("geometric", 5.0, 1, c["max_len"]))


def _drifts(c):
    return c["ttl"] < 1000


def _ring_len(c):
    return 2 * c["ttl"] if _drifts(c) else 4


def _zipf_ranks(n, universe, s, gen):
    """n ranks in [1, universe] with density r^-s (inverse of the continuous law, rounded)."""
    u = torch.rand(n, dtype=torch.float64, device="cuda", generator=gen)
    a, b = 0.5, universe + 0.5
    if abs(s - 1.0) < 1e-6:
        x = a * torch.exp(u * math.log(b / a))
    else:
        lo, hi = a ** (1 - s), b ** (1 - s)
        x = (lo + u * (hi - lo)).pow(1.0 / (1 - s))
    return torch.floor(x + 0.5).to(torch.int64).clamp_(1, universe)


def _ids(ranks, salt):
    ids = wl.splitmix64_torch(ranks ^ salt)
    return torch.where(ids == -1, torch.full_like(ids, -2), ids)


def _batch_ids(c, n, salt, k, gen):
    """The IDs of batch k of the ring; with `new`, part of the ranks carry an identity that only this batch has."""
    ranks = _zipf_ranks(n, UNIVERSE * c["rows"], c["zipf"], gen)
    ids = _ids(ranks, salt)
    if c["new"] > 0:
        mark = wl.splitmix64_torch(ranks * 0x2545F4914F6CDD1D + (k + 1)) & 0xFFFFF
        ids = torch.where(mark < int(c["new"] * 0x100000), _ids(ranks, salt ^ (0x51ED2701 * (k + 1))), ids)
    return ids


def _offsets(c, gen):
    if c["lens"] == "uniform":
        n = torch.randint(1, c["max_len"] + 1, (c["bags"],), device="cuda", generator=gen)
    else:
        u = torch.rand(c["bags"], dtype=torch.float64, device="cuda", generator=gen)
        n = (torch.floor(torch.log1p(-u) / math.log(0.8)) + 1).clamp_(1, c["max_len"]).to(torch.int64)
    off = torch.zeros(c["bags"] + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(n, 0, out=off[1:])
    return off


def _one_table(c, seed):
    """A table as a long-running job has it, a ring of batches, gradients and the buffer the pooled rows go to."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 1000003 + 17)
    salt = wl._signed64(int(wl.splitmix64(np.array([int(seed) + 1], dtype=np.uint64))[0]))
    off = _offsets(c, gen)
    n = int(off[-1])
    ring = [(_batch_ids(c, n, salt, k, gen), off) for k in range(_ring_len(c))]
    more = {"sketch_depth": 4, "sketch_width": 2 << c["rows"].bit_length()} if c["sketch"] else {}
    table = mb.MonoTable(c["rows"], c["dim"], c["threshold"], c["ttl"], lr=0.05, init_scale=0.01, seed=int(seed) & 0xFFFF,
                         max_ids=n, max_bags=c["bags"], **more)
    if not _drifts(c):
        half = c["rows"] // 2
        ranks = torch.randperm(2 * half, device="cuda", generator=gen) + 1
        owns = (ranks <= half).to(torch.uint8)
        waiting = torch.randint(1, max(c["threshold"], 2), ranks.shape, device="cuda", generator=gen)
        count = torch.where(owns > 0, torch.full_like(waiting, c["threshold"]), waiting).to(torch.int32)
        if c["threshold"] == 1:                 # every ID that is tracked owns a row: nobody is on probation
            keep = owns > 0
            ranks, owns, count = ranks[keep], owns[keep], count[keep]
        mb.mono_import(table.handle, _ids(ranks, salt), count, torch.zeros_like(ranks), owns, None, None, ranks.numel())
    grad = torch.randn((c["bags"], c["dim"]), device="cuda", generator=gen).mul_(0.01)
    out = torch.empty((c["bags"], c["dim"]), device="cuda")
    return {"table": table, "ring": ring, "grad": grad, "out": out, "n": n}


def _tables_of(c):
    """The single-table cases of a grouped one: uneven batches, mixed dims up to the case's own."""
    dims = [d for d in GROUP_DIMS if d < c["dim"]] + [c["dim"]]
    return [dict(c, bags=max(1, c["bags"] >> (t % 4)), dim=dims[t % len(dims)]) for t in range(c["tables"])]


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "group":
        parts = [_one_table(p, int(seed) * 977 + t) for t, p in enumerate(_tables_of(c))]
        state = {"handles": [p["table"].handle for p in parts], "tables": [p["table"] for p in parts],
                 "ids": [[p["ring"][k][0] for p in parts] for k in range(_ring_len(c))],
                 "off": [p["ring"][0][1] for p in parts], "grad": [p["grad"] for p in parts],
                 "out": [p["out"] for p in parts], "case": c, "k": 0, "now": 1}
        mb.mono_group_prepare_push(state["handles"], state["ids"][0], state["off"])
        mb.mono_group_lookup_pool(state["handles"], state["ids"][0], state["off"], state["out"])
        return state
    state = dict(_one_table(c, seed), case=c, k=0, now=1)
    ring, h, n, bags = state["ring"], state["table"].handle, state["n"], c["bags"]
    if kind == "push":
        state["distinct"] = [torch.unique(ids) for ids, _ in ring]
        state["each"] = [torch.arange(u.numel() + 1, device="cuda") for u in state["distinct"]]
        # (room for every ID of a batch to be distinct, whatever the lengths drawn; what a batch does not fill stays zero)
        most = max(n, int(1.05 * bags * _mean_len(c)) + 4096)
        state["rows_out"] = torch.zeros((most, c["dim"]), device="cuda")
        mb.mono_reserve(h, most, most)
    elif kind == "host":
        state["ring"] = [(ids.cpu().pin_memory(), off.cpu().pin_memory()) for ids, off in ring]
        state["grad"] = state["grad"].cpu().pin_memory()
        state["out"] = torch.empty((bags, c["dim"])).pin_memory()
        mb.mono_lookup_pool_host(h, state["ring"][0][0], n, state["ring"][0][1], bags, state["out"])
        mb.mono_fence(h)
    elif kind == "train":
        mb.mono_prepare_push(h, ring[0][0], n, ring[0][1], bags)
        mb.mono_group_ahead(h, ring[1][0], n, ring[1][1], bags)
        mb.mono_lookup_pool(h, ring[0][0], n, ring[0][1], bags, state["out"])
        if _drifts(c):
            for _ in range(2 * len(ring)):      # past the first expiries
                run(state)
    return state


# ---- one pass ---------------------------------------------------------------

def run(state):
    return {"pull": _pull, "train": _train, "push": _push, "group": _group, "host": _host}[state["case"]["kind"]](state)


def _turn(state):
    """This pass's batch number, the next one's, the one after that, and the time."""
    k, now, m = state["k"], state["now"], len(state.get("ring") or state["ids"])
    state["k"], state["now"] = (k + 1) % m, now + 1
    return k, (k + 1) % m, (k + 2) % m, now


def _pull(state):
    k, _, _, _ = _turn(state)
    ids, off = state["ring"][k]
    return state["table"].lookup_pool(ids, off, out=state["out"])


def _train(state):
    k, nxt, after, now = _turn(state)
    h, ring, n, bags = state["table"].handle, state["ring"], state["n"], state["case"]["bags"]
    mb.mono_apply_grads(h, ring[k][0], n, ring[k][1], bags, state["grad"], now)
    if _drifts(state["case"]):
        mb.mono_expire(h, now)
    else:
        mb.mono_expire_slice(h, now, now % 32, 32)
    mb.mono_prepare_push(h, ring[nxt][0], n, ring[nxt][1], bags)
    mb.mono_group_ahead(h, ring[after][0], n, ring[after][1], bags)
    mb.mono_lookup_pool(h, ring[nxt][0], n, ring[nxt][1], bags, state["out"])
    return state["out"]


def _push(state):
    k, _, _, now = _turn(state)
    ids, off = state["ring"][k]
    distinct = state["distinct"][k]
    state["table"].apply_grads(ids, off, state["grad"], now)
    state["table"].lookup_pool(distinct, state["each"][k], out=state["rows_out"])
    return state["rows_out"]


def _group(state):
    k, nxt, _, now = _turn(state)
    h, ids, off = state["handles"], state["ids"], state["off"]
    mb.mono_group_apply_grads(h, ids[k], off, state["grad"], now)
    mb.mono_expire(h[now % len(h)], now)
    mb.mono_group_prepare_push(h, ids[nxt], off)
    mb.mono_group_lookup_pool(h, ids[nxt], off, state["out"])
    return state["out"]


def _host(state):
    k, nxt, _, now = _turn(state)
    h, ring, n, bags = state["table"].handle, state["ring"], state["n"], state["case"]["bags"]
    mb.mono_apply_grads_host(h, ring[k][0], n, ring[k][1], bags, state["grad"], now)
    mb.mono_lookup_pool_host(h, ring[nxt][0], n, ring[nxt][1], bags, state["out"])
    mb.mono_fence(h)
    return state["out"]


# ---- what a pass cannot do without -------------------------------------------

def _expected(c):
    """Expected IDs, distinct IDs and distinct IDs with a row in one batch, under the Zipf law of the stream."""
    n = c["bags"] * _mean_len(c)
    v = UNIVERSE * c["rows"]
    edge = np.unique(np.floor(np.geomspace(1, v + 1, 4000)).astype(np.int64))
    width = np.diff(edge).astype(np.float64)
    rank = (edge[:-1] + edge[1:] - 1) / 2.0
    p = rank ** -c["zipf"]
    lam = n * p / (p * width).sum()
    seen = width * -np.expm1(-lam)
    if c["kind"] == "pull":
        owns = rank <= c["rows"] // 2
    elif _drifts(c):
        owns = lam * (c["ttl"] + 1) >= c["threshold"]
    else:
        owns = np.ones_like(rank, dtype=bool)
    return n, float(seen.sum()), float(seen[owns].sum())


def work(case):
    if case["kind"] == "group":
        each = [work(dict(p, kind="train")) for p in _tables_of(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    c, d, b = case, case["dim"], case["bags"]
    n, u, ur = _expected(c)
    ids = 8 * (b + 1) + 8 * n
    keys = 32 * u                                            # a key cell's sector for each distinct ID
    pull = 4 * d * ur + 4 * d * b                            # each row once, the pooled rows
    push = keys + 4 * d * b + 16 * d * ur                    # the cells written, the gradients, rows and accumulators in and out
    if c["kind"] == "pull":
        return {"bytes": ids + keys + pull, "flops": d * n}
    if c["kind"] == "push":                                  # and the distinct IDs' rows read back: ID, offset, cell, row in and out
        return {"bytes": ids + keys + push + u * (8 + 8 + 32) + 8 * d * ur, "flops": d * n + 8 * d * ur}
    return {"bytes": ids + keys + pull + push, "flops": 2 * d * n + 8 * d * ur}


def tolerance(case):
    # sums of fp32 values in a fixed order, gradient sums in fp64 rounded once, IEEE operations elsewhere
    return {"rel": 1e-5}
