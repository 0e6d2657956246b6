"""Edges of the launch rules: the pooling kernels' tiles and vector widths, the parts of long
segments and the tree their partial sums go up, the host-buffer staging taken in turn."""
import numpy as np
import pytest
import torch

from oracle import mono_oracle as mo
from paper_2209_07663_b200 import binding as mb
from paper_2209_07663_b200 import workload as wl
from tests.parity import assert_audit_ok, assert_state_equal, assert_vectors_close

pytestmark = pytest.mark.gpu
f32 = np.float32


def filled(dim, n=4000, capacity=4096):
    """A table whose n IDs own rows of known values."""
    rng = np.random.default_rng(dim)
    ids = wl.splitmix64(np.arange(1, n + 1, dtype=np.uint64))
    w = rng.standard_normal((n, dim)).astype(f32)
    t = mb.MonoTable(capacity, dim, 1, 0, key_cells=1 << 14)
    t.import_entries(ids, np.ones(n, np.uint32), np.zeros(n, np.int64), np.ones(n, np.uint8), w, np.zeros_like(w))
    return t, ids, w


def pulls(t, ids, w, lens, rng, offset_floats=0, break_at=None):
    """Pull bags of these lengths (some IDs unknown), announced and not; compare with a sum in double."""
    dim, n = t.dim, len(ids)
    total = int(np.sum(lens))
    pick = rng.integers(0, n + n // 8, total)                      # beyond n: an ID the table does not know
    flat = np.where(pick < n, ids[np.minimum(pick, n - 1)], np.uint64(1) + pick.astype(np.uint64)).astype(np.uint64)
    off = np.zeros(len(lens) + 1, np.int64)
    off[1:] = np.cumsum(lens)
    rows = np.where((pick < n)[:, None], w[np.minimum(pick, n - 1)], 0).astype(np.float64)
    want = np.stack([rows[off[b]:off[b + 1]].sum(axis=0) if lens[b] else np.zeros(dim) for b in range(len(lens))])
    if break_at is not None:                                       # one bag malformed: it and the next read as empty or as they stand
        off[break_at + 1] = off[break_at] - 1
        want[break_at] = 0
        lo, hi = off[break_at + 1], off[break_at + 2]
        want[break_at + 1] = rows[lo:hi].sum(axis=0) if lo >= 0 else 0
    d_ids, d_off = torch.from_numpy(flat.view(np.int64)).cuda(), torch.from_numpy(off).cuda()
    store = torch.full((len(lens) * dim + 8,), float("nan"), device="cuda")
    out = store[offset_floats:offset_floats + len(lens) * dim]
    for announced in (False, True):
        out.fill_(float("nan"))
        if announced:
            mb.mono_prepare_push(t.handle, d_ids, total, d_off, len(lens))
        mb.mono_lookup_pool(t.handle, d_ids, total, d_off, len(lens), out)
        assert_vectors_close(out.cpu().numpy().reshape(-1, dim), want.astype(f32), f"dim {dim}, announced {announced}")


@pytest.mark.parametrize("dim", [4, 12, 64, 100, 128, 132, 136, 200, 512, 520])
def test_pull_at_every_width_and_alignment(dim):
    t, ids, w = filled(dim)
    rng = np.random.default_rng(1)
    for shift in (0, 4):                                           # 32-byte and only 16-byte aligned output
        pulls(t, ids, w, rng.integers(0, 20, 700), rng, offset_floats=shift)
    assert t.status()["error_bits"] == 0


@pytest.mark.parametrize("lens", [
    [1], [0], [1024], [1025], [5000], [0] * 9 + [33], [1] * 256, [1] * 257, [2] * 8,
    [31, 32, 33, 63, 64, 65] * 50, [1] * 300 + [1023] + [1] * 300, [700, 400] * 20, list(range(40)) * 30,
], ids=lambda v: f"{len(v)}x{max(v)}")
def test_pull_at_the_edges_of_tiles(lens):
    for dim in (16, 200):
        t, ids, w = filled(dim)
        pulls(t, ids, w, np.array(lens), np.random.default_rng(2))
        assert t.status()["error_bits"] == 0


@pytest.mark.parametrize("lens", [[3] * 400, [700, 400] * 20])
def test_pull_with_a_malformed_bag_in_a_tile(lens):
    t, ids, w = filled(32)
    pulls(t, ids, w, np.array(lens), np.random.default_rng(3), break_at=5)
    assert t.status()["error_bits"] == mb.MONO_DEV_BAD_OFFSETS


# multiplicities at the edges of parts (64) and of the levels of their tree (16, 256 and 4096 parts); the second
# batch has more parts than get a warp each, the third more gradients than are left in the order they come
@pytest.mark.parametrize("mult,dim,n_bags", [
    ([63, 64, 65, 128, 1024, 1025, 1088, 16384, 16385], 32, 3000),
    ([300000, 64 * 256 + 1, 65, 1], 8, 20000),
    ([16385, 1024, 65, 64], 520, 40000),
])
@pytest.mark.parametrize("announced", [False, True])
def test_long_segments_at_the_edges_of_the_tree(mult, dim, n_bags, announced):
    kw = dict(init_scale=0.05, seed=9)
    gpu, cpu = mb.MonoTable(64, dim, 1, 0, **kw), mo.OracleTable(64, dim, 1, 0, **kw)
    rng = np.random.default_rng(4)
    ids = rng.permutation(np.repeat(wl.splitmix64(np.arange(len(mult), dtype=np.uint64)), mult))
    cuts = np.sort(rng.integers(0, ids.size + 1, n_bags - 1))
    off = np.concatenate([[0], cuts, [ids.size]]).astype(np.int64)
    for now in range(2):                                           # the second push finds counters and set as the first left them
        grad = (rng.standard_normal((n_bags, dim)) * 0.01).astype(f32)
        d = [torch.from_numpy(x).cuda() for x in (ids.view(np.int64), off, grad)]
        if announced:
            mb.mono_prepare_push(gpu.handle, d[0], ids.size, d[1], n_bags)
        mb.mono_apply_grads(gpu.handle, d[0], ids.size, d[1], n_bags, d[2], now)
        cpu.apply_grads(ids, off, grad, now)
        assert_state_equal(gpu, cpu, f"push {now}")
    assert_audit_ok(gpu)
    assert gpu.status()["error_bits"] == 0


def test_distinct_ids_fill_the_first_tier_of_the_call_set():
    """Batches of distinct IDs only: the primary tier has a slot for each, and what does not find one near
    its place overflows; both tiers have to be empty again for the next push."""
    kw = dict(init_scale=0.05, seed=3)
    gpu, cpu = mb.MonoTable(1 << 14, 16, 1, 0, max_ids=8192, **kw), mo.OracleTable(1 << 14, 16, 1, 0, **kw)
    rng = np.random.default_rng(5)
    for now in range(3):
        ids = wl.splitmix64(np.arange(now * 1000, now * 1000 + 8192, dtype=np.uint64))
        off = np.arange(0, 8193, 4, dtype=np.int64)
        grad = (rng.standard_normal((2048, 16)) * 0.01).astype(f32)
        gpu.apply_grads(ids, off, grad, now)
        cpu.apply_grads(ids, off, grad, now)
    assert_state_equal(gpu, cpu)


def test_host_buffers_are_staged_in_turn():
    """Pulls without a push, pushes of another batch, and several steps in flight: every batch has to be read from
    the buffers it was staged in."""
    cfg = wl.scaled(wl.CONFIGS["tiny"], n_examples=128, filter_threshold=1)
    kw = dict(lr=cfg.lr, eps=cfg.eps, init_scale=cfg.init_scale, seed=cfg.seed)
    gpu = mb.MonoTable(cfg.capacity, cfg.dim, 1, 0, key_cells=cfg.key_cells, max_ids=4096, max_bags=cfg.n_bags, **kw)
    cpu = mo.OracleTable(cfg.capacity, cfg.dim, 1, 0, **kw)
    steps = [wl.Stream(cfg).step(t) for t in range(8)]
    host = [[torch.from_numpy(x).pin_memory() for x in (s.ids.view(np.int64), s.offsets, s.grad_pooled)] for s in steps]
    outs, wants = [], []

    def pull(k):
        outs.append(torch.full((cfg.n_bags, cfg.dim), float("nan")).pin_memory())
        mb.mono_lookup_pool_host(gpu.handle, host[k][0], host[k][0].numel(), host[k][1], cfg.n_bags, outs[-1])
        wants.append(cpu.lookup_pool(steps[k].ids, steps[k].offsets))

    def push(k, now):
        mb.mono_apply_grads_host(gpu.handle, host[k][0], host[k][0].numel(), host[k][1], cfg.n_bags, host[k][2], now)
        cpu.apply_grads(steps[k].ids, steps[k].offsets, steps[k].grad_pooled, now)

    push(0, 0)
    for now in range(1, 4):
        pull(now), pull(now + 1), pull(now)
        push(now, 2 * now)
        push(now + 4, 2 * now + 1)
    mb.mono_fence(gpu.handle)
    torch.cuda.synchronize()
    for k, (got, want) in enumerate(zip(outs, wants)):
        assert_vectors_close(got.numpy(), want, f"pull {k}")
    assert_state_equal(gpu, cpu)


@pytest.mark.parametrize("dim", [16, 64])
@pytest.mark.parametrize("repeats", [1, 64])
def test_look_ups_find_entries_wherever_they_sit(dim, repeats):
    """A key store at load 0.97: entries in their preferred cell, elsewhere in either bucket, and in the overflow
    stash; unknown IDs too.  One batch is one wave of blocks, the other several."""
    n = 3970
    ids = wl.splitmix64(np.arange(1, n + 1, dtype=np.uint64))
    w = np.random.default_rng(7).standard_normal((n, dim)).astype(f32)
    t = mb.MonoTable(4096, dim, 1, 0, key_cells=4096, seed=5)
    t.import_entries(ids, np.ones(n, np.uint32), np.zeros(n, np.int64), np.ones(n, np.uint8), w, np.zeros_like(w))
    assert t.status()["error_bits"] == 0 and t.status()["n_evictions_total"] > 0
    known = np.tile(ids, repeats)
    flat = np.concatenate([known, wl.splitmix64(np.arange(10 ** 6, 10 ** 6 + 500, dtype=np.uint64))])
    want = torch.from_numpy(np.concatenate([np.tile(w, (repeats, 1)), np.zeros((500, dim), f32)])).cuda()
    d_ids = torch.from_numpy(flat.view(np.int64)).cuda()
    d_off = torch.arange(flat.size + 1, device="cuda")
    for announced in (False, True):
        out = torch.full((flat.size, dim), float("nan"), device="cuda")
        if announced:
            mb.mono_prepare_push(t.handle, d_ids, flat.size, d_off, flat.size)
        mb.mono_lookup_pool(t.handle, d_ids, flat.size, d_off, flat.size, out)
        assert torch.equal(out, want), announced


def test_batches_of_many_sizes_share_one_reservation():
    """The primary tier follows the batch: sizes at its powers of two, up and down, all-distinct and repeated, on every
    path a batch can come, each grouped while another of a different size is still on its way."""
    sizes = [1 << 17, 1, 1023, 1024, 1025, 2048, 2049, 40000, 1 << 16, (1 << 16) + 1, 7, 100000, 3, 1 << 17]
    kw = dict(init_scale=0.05, seed=3)
    gpu = mb.MonoTable(1 << 19, 8, 1, 0, max_ids=1 << 17, max_bags=1 << 16, **kw)
    cpu = mo.OracleTable(1 << 19, 8, 1, 0, **kw)
    rng = np.random.default_rng(6)

    def batch(k, n):
        ranks = np.arange(n) + 1000 * k if k % 2 == 0 else rng.integers(0, max(n // 3, 1), n)
        off = np.append(np.arange(0, n, 3), n).astype(np.int64)
        ids = wl.splitmix64(ranks.astype(np.uint64))
        grad = (rng.standard_normal((off.size - 1, 8)) * 0.01).astype(f32)
        return ids, off, grad, [torch.from_numpy(x).cuda() for x in (ids.view(np.int64), off, grad)]

    batches = [batch(k, n) for k, n in enumerate(sizes)]
    for k, (ids, off, grad, d) in enumerate(batches):
        bags = off.size - 1
        if k % 3:                                                  # (two of three: announced, half of those pulled)
            mb.mono_prepare_push(gpu.handle, d[0], ids.size, d[1], bags)
            nxt = batches[(k + 1) % len(batches)]
            mb.mono_group_ahead(gpu.handle, nxt[3][0], nxt[0].size, nxt[3][1], nxt[1].size - 1)
        if k % 3 == 1:
            out = torch.full((bags, 8), float("nan"), device="cuda")
            mb.mono_lookup_pool(gpu.handle, d[0], ids.size, d[1], bags, out)
            assert_vectors_close(out.cpu().numpy(), cpu.lookup_pool(ids, off), f"pull {k}")
        if k == 8:
            mb.mono_group_apply_grads([gpu.handle], [d[0]], [d[1]], [d[2]], k)
        else:
            mb.mono_apply_grads(gpu.handle, d[0], ids.size, d[1], bags, d[2], k)
        cpu.apply_grads(ids, off, grad, k)
    assert_state_equal(gpu, cpu)
    assert_audit_ok(gpu)
    assert gpu.status()["scratch_reallocs"] == 0 and gpu.status()["error_bits"] == 0


def test_a_small_push_costs_the_same_in_a_large_reservation():
    """Emptying the per-call set goes by the batch: wiping a tier sized for 2^21 IDs with the few blocks of 168 made the
    row updates 285 us, fifteen times what they take with a tier of the batch's own size (so three is far from either)."""
    ids = torch.from_numpy(wl.splitmix64(np.arange(168, dtype=np.uint64)).view(np.int64)).cuda()
    off, grad = torch.arange(169, device="cuda"), torch.zeros((168, 32), device="cuda")
    us = []
    for reserved in (1024, 1 << 21):
        t = mb.MonoTable(1 << 12, 32, 1, 0, max_ids=reserved, max_bags=1024)
        best = float("inf")
        mb.mono_timing_enable(t.handle, True)
        for now in range(20):
            mb.mono_apply_grads(t.handle, ids, 168, off, 168, grad, now)
            best = min(best, mb.mono_timing_read(t.handle, reset=True)["kernels"]["update_rows"]["ms"])
        us.append(best * 1e3)
        t.close()
    assert us[1] < 3 * us[0], us


@pytest.mark.parametrize("n, key_cells", [(60, 64), (900, 1 << 12), (4000, 1 << 12), (4000, 1 << 23), (3 << 20, 1 << 23)])
@pytest.mark.parametrize("slices", [1, 3])
def test_sweeps_of_sparse_and_dense_key_stores(n, key_cells, slices):
    """Blocks with one round of buckets and with several, few buckets to open (listed over several rounds) and nearly all;
    entries of all ages swept three times, so that the second and third go by the records that the one before left."""
    rng = np.random.default_rng(n)
    ttl, capacity = 10, n + 5
    ids = wl.splitmix64(np.arange(1, n + 1, dtype=np.uint64))
    seen = rng.integers(0, 40, n)
    owns = (rng.random(n) < 0.6).astype(np.uint8)
    t = mb.MonoTable(capacity, 4, 3, ttl, key_cells=key_cells)
    t.import_entries(ids, np.where(owns, 3, 1).astype(np.uint32), seen.astype(np.int64), owns, None, None)
    assert t.status()["n_tracked"] == n
    for now in (20, 21, 45):
        for k in range(slices):
            mb.mono_expire_slice(t.handle, now, k, slices)
        stay = now - seen <= ttl
        st = t.status()
        assert (st["n_tracked"], st["n_resident"], st["n_expired_total"]) == (stay.sum(), (stay & (owns > 0)).sum(), n - stay.sum())
        assert_audit_ok(t, f"now {now}")
        got = t.export(rows=False)
        order = np.argsort(ids[stay])
        assert (got["ids"] == ids[stay][order]).all() and (got["last_seen"] == seen[stay][order]).all()
    assert t.status()["error_bits"] == 0
    t.close()


@pytest.mark.parametrize("announced", [False, True])
@pytest.mark.parametrize("imported_at", [0, 40])
def test_times_of_ids_that_own_rows(announced, imported_at):
    """Their exact time is kept with the row, their cell's is a bound: pushes that leave the cell alone, that have to
    mark it again after an export, and that come before the time in it (imported at 40); sweeps that open buckets for
    cells whose rows were renewed; a snapshot, a rehash."""
    n, ttl, dim = 300, 5, 4
    ids = wl.splitmix64(np.arange(1, n + 1, dtype=np.uint64))
    t = mb.MonoTable(512, dim, 1, ttl, key_cells=512)
    t.import_entries(ids, np.ones(n, np.uint32), np.full(n, imported_at, np.int64), np.ones(n, np.uint8), None, None)
    last = np.full(n, imported_at)

    def check(what):
        got = t.export(rows=False)
        order = np.argsort(ids[last >= 0])
        assert (got["ids"] == ids[last >= 0][order]).all(), what
        assert (got["last_seen"] == last[last >= 0][order]).all(), what
        d = torch.from_numpy(ids.view(np.int64)).cuda()
        seen = torch.empty(n, dtype=torch.int64, device="cuda")
        mb.mono_probe(t.handle, d, n, None, None, seen)
        assert (seen.cpu().numpy() == last).all(), what
        assert_audit_ok(t, what)

    def push(which, now):
        d = torch.from_numpy(ids[which].view(np.int64)).cuda()
        off = torch.arange(d.numel() + 1, device="cuda")
        if announced:
            mb.mono_prepare_push(t.handle, d, d.numel(), off, d.numel())
        mb.mono_apply_grads(t.handle, d, d.numel(), off, d.numel(), torch.zeros((d.numel(), dim), device="cuda"), now)
        last[which] = now

    k = np.arange(n)
    push(k % 3 == 0, 1)
    push(k % 3 == 0, 2)
    push(k % 2 == 0, 4)
    check("pushed")
    assert t.export_touched()["found"] == int(((k % 3 == 0) | (k % 2 == 0)).sum())
    push(k % 5 == 0, 5)
    assert set(t.export_touched()["ids"]) == set(ids[k % 5 == 0])
    mb.mono_snapshot_save(t.handle)
    kept = last.copy()
    push(k % 4 == 0, 6)
    check("pushed again")
    mb.mono_snapshot_restore(t.handle)
    last[:] = kept
    check("restored")
    mb.mono_rehash(t.handle, 1024, 9)
    check("rehashed")
    for now in (6, 8, 10, 11):
        t.expire(now)
        last[(last >= 0) & (now - last > ttl)] = -1
        check(f"swept at {now}")
        if now == 8:
            push((k % 7 == 0) & (last >= 0), 9)
    assert (last >= 0).any() and (last < 0).any()
    assert t.status()["error_bits"] == 0


@pytest.mark.parametrize("path", ["plain", "announced", "grouped"])
@pytest.mark.parametrize("key_cells", [512, 1 << 13])
def test_an_entry_pushed_before_its_imported_time_expires_by_the_push(path, key_cells):
    """Entries imported at a later time than the pushes that follow: a push writes the earlier time, and the bucket's
    record, which is what the sweep goes by, may not stay at the later one."""
    n, ttl, dim = 400, 5, 4
    ids = wl.splitmix64(np.arange(1, n + 1, dtype=np.uint64))
    owns = np.arange(n) % 2
    t = mb.MonoTable(512, dim, 4, ttl, key_cells=key_cells)
    t.import_entries(ids, np.where(owns, 4, 1).astype(np.uint32), np.full(n, 40, np.int64), owns.astype(np.uint8), None, None)
    last = np.full(n, 40)
    for which, now in ((np.arange(n) % 3 == 0, 1), (np.arange(n) % 5 == 0, 10)):
        d = torch.from_numpy(ids[which].view(np.int64)).cuda()
        off, grad = torch.arange(d.numel() + 1, device="cuda"), torch.zeros((d.numel(), dim), device="cuda")
        if path == "announced":
            mb.mono_prepare_push(t.handle, d, d.numel(), off, d.numel())
        if path == "grouped":
            mb.mono_group_apply_grads([t.handle], [d], [off], [grad], now)
        else:
            mb.mono_apply_grads(t.handle, d, d.numel(), off, d.numel(), grad, now)
        last[which] = now
        assert_audit_ok(t, f"pushed at {now}")
    for now in (12, 20, 50):
        t.expire(now)
        stay = now - last <= ttl
        got = t.export(rows=False)
        order = np.argsort(ids[stay])
        assert (got["ids"] == ids[stay][order]).all() and (got["last_seen"] == last[stay][order]).all(), now
        assert_audit_ok(t, f"swept at {now}")
    assert t.status()["error_bits"] == 0


@pytest.mark.parametrize("grouped", [False, True])
@pytest.mark.parametrize("dim, n_bags", [(16, 300), (512, 34000)])
def test_counters_start_afresh_with_every_batch(dim, n_bags, grouped):
    """Batches announced, grouped ahead and forgotten again, some with a malformed bag, between batches that are pushed: what
    was counted for the forgotten ones (IDs, parts and their order, the malformed bag) is in no later one.  34 000
    bags of 512 columns are beyond 64 MB, so their parts are put in order."""
    kw = dict(init_scale=0.05, seed=6)
    gpu, cpu = mb.MonoTable(1 << 12, dim, 2, 0, **kw), mo.OracleTable(1 << 12, dim, 2, 0, **kw)
    rng = np.random.default_rng(dim)
    h, known, sums = gpu.handle, set(), np.zeros(3, np.int64)

    def batch(spoilt=False):
        n = 3 * n_bags
        hot = np.repeat(rng.permutation(50)[:3], (70, n // 8, n // 4))
        ids = np.concatenate([hot, rng.integers(50, 3000, n - hot.size)])
        ids = wl.splitmix64(rng.permutation(ids).astype(np.uint64))
        off = np.append(np.arange(0, ids.size, 3), ids.size).astype(np.int64)
        grad = (rng.standard_normal((off.size - 1, dim)) * 0.01).astype(f32)
        if spoilt:
            off[7] = off[6] - 2
        return ids, off, grad, [torch.from_numpy(x).cuda() for x in (ids.view(np.int64), off, grad)]

    def announce(b):
        if grouped:
            mb.mono_group_prepare_push([h], [b[3][0]], [b[3][1]])
        else:
            mb.mono_prepare_push(h, b[3][0], b[0].size, b[3][1], b[1].size - 1)

    def ahead(b):
        mb.mono_group_ahead(h, b[3][0], b[0].size, b[3][1], b[1].size - 1)

    def push(b, now):
        if grouped:
            mb.mono_group_apply_grads([h], [b[3][0]], [b[3][1]], [b[3][2]], now)
        else:
            mb.mono_apply_grads(h, b[3][0], b[0].size, b[3][1], b[1].size - 1, b[3][2], now)
        cpu.apply_grads(b[0], b[1], b[2], now)
        distinct = set(b[0].tolist())
        sums[:] += (b[0].size, len(distinct), len(distinct - known))
        known.update(distinct)
        st = gpu.status()
        assert [st[k] for k in ("sum_ids", "sum_unique", "sum_new")] == sums.tolist(), now

    for now in range(6):
        good = batch()
        if now == 1:
            announce(batch())                                      # given up for another announcement
            announce(good)
        elif now == 2:
            announce(batch())                                      # given up by a push
        elif now == 3:
            ahead(batch(spoilt=True))                              # never taken over
            ahead(good)
            announce(good)
        elif now == 4:
            announce(batch())
            mb.mono_export_touched(h, None, None, 0)               # forgets it
        elif now == 5:
            announce(batch(spoilt=True))
            assert gpu.status()["error_bits"] == mb.MONO_DEV_BAD_OFFSETS
            mb.mono_clear_errors(h)
        push(good, now)
        assert gpu.status()["error_bits"] == 0, now
    push(batch(), 6)
    assert_state_equal(gpu, cpu)
    assert_audit_ok(gpu)
    assert gpu.status()["error_bits"] == 0


@pytest.mark.parametrize("n_tables", [1, 2, 31, 32, 33, 65, 150])
def test_grouped_calls_find_every_block_its_table(n_tables):
    """Numbers of tables around those that a warp searches at once; batches of very different size, every fifth empty.
    Against the single-table calls on tables of their own."""
    rng = np.random.default_rng(n_tables)
    dims = [4, 20, 64, 128, 132]
    pair, batch = [[], []], []
    for i in range(n_tables):
        for side in pair:
            side.append(mb.MonoTable(256, dims[i % 5], 1, 0, key_cells=1024, init_scale=0.1, seed=i))
        bags = 0 if i % 5 == 4 and i else int(rng.integers(1, 60)) if i % 7 else 900
        ids = wl.splitmix64(rng.integers(0, 200, bags * 3).astype(np.uint64))
        grad = (rng.standard_normal((bags, dims[i % 5])) * 0.01).astype(f32)
        batch.append([torch.from_numpy(x).cuda() for x in (ids.view(np.int64), np.arange(0, 3 * bags + 1, 3), grad)])
    ids, off, grad = ([b[k] for b in batch] for k in range(3))
    grouped, single = [[t.handle for t in side] for side in pair]
    for now in range(3):
        out = [torch.full((b[1].numel() - 1, t.dim), float("nan"), device="cuda") for b, t in zip(batch, pair[0])]
        if now:
            mb.mono_group_prepare_push(grouped, ids, off)
        mb.mono_group_lookup_pool(grouped, ids, off, out)
        mb.mono_group_apply_grads(grouped, ids, off, grad, now)
        for i, t in enumerate(single):
            want = torch.zeros_like(out[i])
            bags = off[i].numel() - 1
            mb.mono_lookup_pool(t, ids[i], ids[i].numel(), off[i], bags, want)
            mb.mono_apply_grads(t, ids[i], ids[i].numel(), off[i], bags, grad[i], now)
            assert_vectors_close(out[i].cpu().numpy(), want.cpu().numpy(), f"table {i}, step {now}")
    for g, s in zip(*pair):
        a, b = g.export(), s.export()
        assert (a["ids"] == b["ids"]).all() and (a["count"] == b["count"]).all() and (a["last_seen"] == b["last_seen"]).all()
        assert_vectors_close(a["w"], b["w"], "rows")
        assert_vectors_close(a["acc"], b["acc"], "accumulators")
        assert g.status()["error_bits"] == 0


@pytest.mark.parametrize("dim", [260, 512, 516, 1024])
@pytest.mark.parametrize("announced", [False, True])
def test_grouped_calls_of_the_widest_rows(dim, announced):
    """Rows of more than 256 columns beside narrow ones in one group: segments of 1 to 66 occurrences and long ones, whose
    parts go up one level of the tree and two; long bags and empty ones; pooled to an output aligned to 32 bytes and to 16."""
    pair, batch = [], []
    for k, d in enumerate((dim, 16, dim)):
        kw = dict(init_scale=0.05, seed=k)
        pair.append((mb.MonoTable(512, d, 2, 0, key_cells=2048, **kw), mo.OracleTable(512, d, 2, 0, **kw)))
        rng = np.random.default_rng(dim + k)
        times = np.concatenate([np.arange(1, 67), [200, 1500], np.ones(60, np.int64)])
        ids = rng.permutation(np.repeat(wl.splitmix64(np.arange(1, times.size + 1, dtype=np.uint64)), times))
        off = np.sort(np.concatenate([[0, ids.size], rng.integers(0, ids.size, 400)])).astype(np.int64)
        grad = (rng.standard_normal((off.size - 1, d)) * 0.01).astype(f32)
        batch.append((ids, off, grad))
    h = [g.handle for g, _ in pair]
    ids, off, grad = ([torch.from_numpy(b[k].view(np.int64) if k == 0 else b[k]).cuda() for b in batch] for k in range(3))
    for now in range(3):
        stores = [torch.full((b[2].size + 8,), float("nan"), device="cuda") for b in batch]
        out = [s[4 * (now % 2):][:b[2].size].view(b[2].shape) for s, b in zip(stores, batch)]
        if announced:
            mb.mono_group_prepare_push(h, ids, off)
        mb.mono_group_lookup_pool(h, ids, off, out)
        for (_, cpu), b, o in zip(pair, batch, out):
            assert_vectors_close(o.cpu().numpy(), cpu.lookup_pool(b[0], b[1]), f"step {now}")
        mb.mono_group_apply_grads(h, ids, off, grad, now)
        for (_, cpu), b in zip(pair, batch):
            cpu.apply_grads(*b, now)
    for gpu, cpu in pair:
        assert_state_equal(gpu, cpu)
        assert_audit_ok(gpu)
        assert gpu.status()["error_bits"] == 0


def test_every_launch_of_a_call_is_counted():
    """A grouped step's, the uploads of its descriptors among them, for its first table; the wipes of batches that are
    forgotten."""
    n = 100
    pair = [mb.MonoTable(256, dim, 1, 0, key_cells=1024, max_ids=n, max_bags=n) for dim in (8, 64)]
    h = [t.handle for t in pair]
    ids = [torch.arange(1 + k, n + 1 + k, device="cuda") for k in range(2)]
    off = [torch.arange(n + 1, device="cuda")] * 2
    out = [torch.empty((n, t.dim), device="cuda") for t in pair]

    def counted(table):
        got = mb.mono_timing_read(table, reset=True)
        each = {k: v["launches"] for k, v in got["kernels"].items() if v["launches"]}
        assert got["launches_total"] == sum(each.values())
        return each

    counted(h[0]), counted(h[1])
    mb.mono_group_prepare_push(h, ids, off)
    mb.mono_group_lookup_pool(h, ids, off, out)
    mb.mono_group_apply_grads(h, ids, off, out, 1)
    assert counted(h[1]) == {}
    assert counted(h[0]) == {"group_upload": 3, **dict.fromkeys(("fill_occ_bag", "dedup_tile", "table_lookup", "gather_pool", "table_update", "table_insert", "update_rows"), 1)}
    mb.mono_prepare_push(h[0], ids[0], n, off[0], n)
    mb.mono_prepare_push(h[0], ids[1], n, off[1], n)
    mb.mono_group_ahead(h[0], ids[0], n, off[0], n)
    mb.mono_group_ahead(h[0], ids[1], n, off[1], n)
    assert counted(h[0]) == {"wipe_call_set": 2, "fill_occ_bag": 4, "dedup_tile": 4, "table_lookup": 2}
    for t in pair:
        t.close()


@pytest.mark.parametrize("repeated", [1, 255, 256, 4096, 4097])
@pytest.mark.parametrize("dim", [4, 20, 64, 100, 132])
@pytest.mark.parametrize("grouped", [False, True])
def test_segments_of_every_length_in_small_and_large_numbers(repeated, dim, grouped):
    """IDs that occur 1 to 66 times, so many of them repeated that a warp, or a lane group, takes each; alone and in a
    grouped call."""
    kw = dict(init_scale=0.05, seed=4)
    gpu, cpu = mb.MonoTable(1 << 14, dim, 1, 0, **kw), mo.OracleTable(1 << 14, dim, 1, 0, **kw)
    rng = np.random.default_rng(repeated + dim)
    times = np.concatenate([np.arange(repeated) % 65 + 2, np.ones(50, np.int64)])
    ids = rng.permutation(np.repeat(wl.splitmix64(np.arange(1, times.size + 1, dtype=np.uint64)), times))
    off = np.unique(np.concatenate([[0, ids.size], rng.integers(0, ids.size, ids.size // 3)])).astype(np.int64)
    grad = (rng.standard_normal((off.size - 1, dim)) * 0.01).astype(f32)
    d = [torch.from_numpy(x).cuda() for x in (ids.view(np.int64), off, grad)]
    for now in range(2):
        if grouped:
            mb.mono_group_apply_grads([gpu.handle], [d[0]], [d[1]], [d[2]], now)
        else:
            mb.mono_apply_grads(gpu.handle, d[0], ids.size, d[1], off.size - 1, d[2], now)
        cpu.apply_grads(ids, off, grad, now)
    assert_state_equal(gpu, cpu)
    assert gpu.status()["error_bits"] == 0


@pytest.mark.parametrize("dim", [16, 32, 64, 128, 136, 256])
@pytest.mark.parametrize("bags, mean", [(300, 3), (300, 9), (3000, 40), (16000, 40)])
def test_pulls_of_short_and_long_bags_in_small_and_large_batches(dim, bags, mean):
    """Both sides of the rule that takes more rows in flight: by the mean bag length, by the size of the batch (one tile
    of 850 IDs per SM, four), announced and not; bags of every length up to twice the mean, so every remainder."""
    t, ids, w = filled(dim)
    rng = np.random.default_rng(bags + mean)
    pulls(t, ids, w, rng.integers(0, 2 * mean + 1, bags), rng)
    assert t.status()["error_bits"] == 0
