"""Inputs at the limits of what the loads accept, by the forms that a caller
gets without naming one (candidate lists alone, in a batch, on a server and
without allocations) and bit-packed, against the oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2109_06042_gb300 import instances as I

pytestmark = pytest.mark.gpu

VARIANTS = [("dp", False), ("se", False), ("dp", True), ("se", True)]
TOP = 2**31 - 1  # the largest demand


@pytest.fixture(scope="module")
def mhs():
    from paper_2109_06042_gb300 import build
    build.build()
    from paper_2109_06042_gb300 import mhs as M
    return M


def _same(got, ref, ctx=""):
    for key in ("vertices", "edges", "demands"):
        assert got[key].tolist() == ref[key].tolist(), (key, ctx)
    assert got["k"] == ref["k"] and got["rounds"] == ref["rounds"], ctx


def _dev(*arrays):
    import torch
    return [torch.from_numpy(np.ascontiguousarray(a, np.int32)).cuda() for a in arrays]


def _noalloc(mhs, inst, ref, ctx=""):
    import torch
    av = torch.full((max(inst.n, 1),), 7, dtype=torch.uint8, device="cuda")
    ae = torch.full((max(inst.m, 1),), 7, dtype=torch.uint8, device="cuda")
    d = _dev(inst.edge_ptr, np.append(inst.edge_vtx, 0), inst.demand)
    assert mhs.kernelize_noalloc(inst.n, inst.m, *d, inst.nnz, av, ae) == ref["rounds"], ctx
    assert torch.nonzero(av[:inst.n]).flatten().tolist() == ref["vertices"].tolist(), ctx
    assert torch.nonzero(ae[:inst.m]).flatten().tolist() == ref["edges"].tolist(), ctx


def _every_form(mhs, insts, rule="dp", fe=False):
    refs = [O.reduce_variant(i, rule, fe) for i in insts]
    opts = {"rule": rule, "full_edges": fe}
    with mhs.Instance.load_batch(insts, **opts) as h:
        h.kernelize()
        for b, ref in enumerate(refs):
            _same(h.result(b), ref, f"batch {b}")
    with mhs.Server(**opts) as srv:
        tickets = [srv.submit(i) for i in insts]
        for b, t in enumerate(tickets):
            _same(srv.poll(t), refs[b], f"server {b}")
    for b, inst in enumerate(insts):
        _same(mhs.kernelize(inst, **opts), refs[b], f"alone {b}")
        _same(mhs.kernelize(inst, contraction="popcount", **opts), refs[b], f"popcount {b}")
        if rule == "dp" and not fe:
            _noalloc(mhs, inst, refs[b], f"noalloc {b}")


@pytest.mark.parametrize("rule,fe", VARIANTS)
def test_the_largest_demands(mhs, rule, fe):
    """Any demand from 1 to 2^31 - 1 is legal: none stands for a deleted hyperedge."""
    rng = np.random.Generator(np.random.PCG64(31))
    insts = [I.from_edges(2, [[0, 1]], [TOP]),
             I.from_edges(5, [[0, 1], [0, 1, 2], [3, 4], [3], []], [TOP, TOP - 1, TOP, 5, TOP])]
    for s in range(24):
        i = I.tiny_random(s, nmax=16, mmax=16)
        i.demand[:] = rng.choice([TOP, TOP - 1, TOP - 2, 2**30, 2**24 + 1, 1, 2, 3], i.m)
        insts.append(i)
    _every_form(mhs, insts, rule, fe)


@pytest.mark.parametrize("f", [2**30 - 2, 2**30 - 1, 2**30 + 5, TOP])
def test_large_demands_on_a_pair_of_heavy_vertices(mhs, f):
    """The bound that a hyperedge of two vertices of high degree sets is as
    large as its demand; supersets of that demand and below go, others stay."""
    edges = [[0, 1]] + [[0, 1, 2 + k] for k in range(300)] + [[0, 1, 2 + k, 3 + k] for k in range(299)]
    dem = [f] + [f] * 300 + [f - k % 7 for k in range(298)] + [TOP]
    same = I.from_edges(302, edges, dem, k=1)
    dem[0] = f - 3
    _every_form(mhs, [same, I.from_edges(302, edges, dem, k=1)])
    _every_form(mhs, [same], fe=True)


def test_a_barrier_that_times_out_is_an_error(mhs):
    """Every kernel of the candidate lists whose CTAs wait for one that never
    comes gives up and the call says so; the next call is right again."""
    import torch
    inst = I.uniform_random(2000, 4000, 2, 8, 3, 5, seed=9)
    ref = O.reduce(inst)
    d = _dev(inst.edge_ptr, inst.edge_vtx, inst.demand)

    def fails(call):
        mhs.selftest_team_wait(1_000_000)
        try:
            with pytest.raises(mhs.MhsError) as ei:
                call()
        finally:
            mhs.selftest_team_wait(0)
        assert ei.value.status == mhs.MHS_EDEVICE

    fails(lambda: mhs.Instance.load(inst))
    fails(lambda: mhs.Instance.load_device(inst.n, inst.m, *d, inst.k))
    fails(lambda: mhs.Instance.load_batch([inst, inst]))
    av, ae = (torch.zeros(x, dtype=torch.uint8, device="cuda") for x in (inst.n, inst.m))
    fails(lambda: mhs.kernelize_noalloc(inst.n, inst.m, *d, inst.nnz, av, ae))
    for insts in ([inst], [inst, inst]):
        for step in ("kernelize", "reduce_round"):
            with mhs.Instance.load_batch(insts) as h:
                fails(getattr(h, step))
                with pytest.raises(mhs.MhsError):
                    h.result()
    for late in ("contract", "end"):
        with mhs.Instance.load(inst) as h:
            h.pass_begin(0)
            if late == "contract":
                mhs.selftest_team_wait(1_000_000)
            h.pass_contract(0, 0, 1)
            mhs.selftest_team_wait(0)
            h.pass_end(0)
            h.pass_begin(1)
            h.pass_contract(1, 0, 1)
            if late == "end":
                fails(lambda: h.pass_end(1))
            else:
                with pytest.raises(mhs.MhsError) as ei:
                    h.pass_end(1)
                assert ei.value.status == mhs.MHS_EDEVICE
    _same(mhs.kernelize(inst), ref)
    _noalloc(mhs, inst, ref)


@pytest.mark.parametrize("rule", ["dp", "se"])
def test_full_lists_of_tasks_and_pairs(mhs, rule):
    """Many more long lists and open pairs than an instance of a batch has room
    for: what finds none is walked and decided in place."""
    rng = np.random.Generator(np.random.PCG64(17))
    insts = []
    for m, n, size in [(700, 14, 7), (400, 24, 20), (300, 70, 60), (500, 20, 10)]:
        edges = [np.sort(rng.choice(n, size + int(rng.integers(0, 2)), replace=False)) for _ in range(m)]
        insts.append(I.from_edges(n, edges, rng.integers(1, 6, m), k=3))
    refs = [O.reduce_variant(i, rule, False) for i in insts]
    for times in (20, 3):  # a CTA for each, teams of CTAs
        with mhs.Instance.load_batch(insts * times, rule=rule) as h:
            h.kernelize()
            assert h.work_stats() == (0, 0)  # by candidate lists
            for b in range(0, len(insts) * times, 7):
                _same(h.result(b), refs[b % len(insts)], b)
    for inst, ref in zip(insts, refs):
        _same(mhs.kernelize(inst, rule=rule), ref)


def _unsorted(n, sizes, seed):
    """Rows in no order, with a few repeats, and the instance that they are."""
    rng = np.random.Generator(np.random.PCG64(seed))
    rows = []
    for s in sizes:
        r = rng.choice(n, s, replace=False)
        rows.append(rng.permutation(np.concatenate([r, r[:rng.integers(0, 4)]])))
    rows += [r[1:] for r in rows[:6]]
    inst = I.from_edges(n, [sorted(set(r.tolist())) for r in rows], rng.integers(1, 5, len(rows)), k=2)
    ptr = np.concatenate([[0], np.cumsum([len(r) for r in rows])])
    return inst, _dev(ptr, np.concatenate(rows), inst.demand)


@pytest.mark.parametrize("n,longest", [(256, 256), (257, 257), (4000, 65), (4000, 1500), (65536, 8100),
                                       (65537, 8100), (70000, 65536), (70000, 65537)])
def test_unsorted_rows_of_any_length(mhs, n, longest):
    """One long row among many short ones: ranked (up to 64 ids), sorted by bytes
    of the id (1, 2 or 3 of them), or (above 65,536) not for this path."""
    inst, d = _unsorted(n, [longest, 63, 64, 65, 128] + [3, 17, 30] * 700, seed=n + longest)
    ref = O.reduce(inst)
    with mhs.Instance.load_device(inst.n, inst.m, *d, inst.k) as h:
        h.kernelize()
        _same(h.result(), ref)
    rows = np.split(d[1].cpu().numpy(), d[0].cpu().numpy()[1:-1])
    host = I.Instance(n=inst.n, m=inst.m, edge_ptr=np.concatenate([[0], np.cumsum(
        [len(set(r.tolist())) for r in rows])]).astype(np.int32), edge_vtx=np.concatenate(
        [np.array(list(dict.fromkeys(r.tolist())), np.int32) for r in rows]),
        demand=inst.demand, k=inst.k)  # host loads refuse repeats
    _same(mhs.kernelize(host), ref)


@pytest.mark.parametrize("length", [64, 65, 4096, 50000])
def test_noalloc_unsorted_rows_with_many_repeats(mhs, length):
    import torch
    rng = np.random.Generator(np.random.PCG64(length))
    n, rows = 4000, [rng.integers(0, 3000, length)] + [rng.choice(4000, 9, replace=False) for _ in range(900)]
    inst = I.from_edges(n, [sorted(set(r.tolist())) for r in rows], rng.integers(1, 4, len(rows)), k=2)
    ref = O.reduce(inst)
    av, ae = (torch.zeros(x, dtype=torch.uint8, device="cuda") for x in (inst.n, inst.m))
    d = _dev(np.concatenate([[0], np.cumsum([len(r) for r in rows])]), np.concatenate(rows), inst.demand)
    assert mhs.kernelize_noalloc(n, inst.m, *d, d[1].numel(), av, ae) == ref["rounds"]
    assert torch.nonzero(av).flatten().tolist() == ref["vertices"].tolist()
    assert torch.nonzero(ae).flatten().tolist() == ref["edges"].tolist()


@pytest.mark.parametrize("heavy", [2, 5, 6, 7, 16, 63, 64, 65, 300])
def test_hyperedges_of_many_heavy_vertices(mhs, heavy):
    """Superseders of demand |e| - 1 .. |e| + 1 over `heavy` vertices of 192
    hyperedges and more, which delete by pairs of them: up to 6 by bounds,
    above by walks, and all by walks where some row has more than 64."""
    rng = np.random.Generator(np.random.PCG64(heavy))
    hubs = heavy + 6
    each = max(1, 260 // hubs)
    edges, dem = [], []
    for q in range(3):
        e = np.sort(rng.choice(hubs, heavy, replace=False)).tolist()
        edges.append(e)
        dem.append(max(1, len(e) - 1 + q))
    for a in range(hubs):
        for b in rng.choice([x for x in range(hubs) if x != a], min(hubs - 1, 40), replace=False):
            for q in range(each):
                edges.append(sorted({a, int(b), hubs + int(rng.integers(0, 900))}))
                dem.append(int(rng.integers(1, 4)))
        for q in range(200):
            edges.append(sorted({a} | {hubs + int(x) for x in rng.integers(0, 900, 2)}))
            dem.append(int(rng.integers(1, 3)))
    inst = I.from_edges(hubs + 900, edges, dem, k=3)
    deg = np.bincount(inst.edge_vtx, minlength=inst.n)
    assert deg[:hubs].min() >= 192
    with mhs.Instance.load(inst) as h:
        h.kernelize()
        assert h.work_stats() == (0, 0)  # by candidate lists
        got = h.result()
    _same(got, O.reduce(inst) if inst.m < 10000 else mhs.kernelize(inst, contraction="popcount"))
    _same(mhs.kernelize(inst, full_edges=True),
          mhs.kernelize(inst, contraction="popcount", full_edges=True))


def test_batch_of_instances_with_and_without_long_rows(mhs):
    """One CTA builds instances of both kinds in turn, below and above the 3,072
    vertices whose degrees it keeps in shared memory; malformed ones are named."""
    import torch
    insts, parts = [], []
    for s, (n, long) in enumerate([(300, 0), (300, 65), (3072, 200), (3073, 0), (3500, 900), (40, 40), (4000, 64)]):
        inst, d = _unsorted(n, [long] * (long > 0) + [5, 9, 16, 17] * 40, seed=s)
        insts.append(inst)
        parts.append([x.cpu().numpy() for x in d])
    refs = [O.reduce(i) for i in insts]
    order = [b % len(insts) for b in range(420)]
    n = np.array([insts[b].n for b in order], np.int32)
    m = np.array([insts[b].m for b in order], np.int32)
    k = np.array([insts[b].k for b in order], np.int64)
    sizes = np.concatenate([np.diff(parts[b][0]) for b in order])
    ptr = torch.from_numpy(np.concatenate([[0], np.cumsum(sizes)])).cuda()
    vtx, dem = _dev(np.concatenate([parts[b][1] for b in order]),
                    np.concatenate([parts[b][2] for b in order]))
    with mhs.Instance.load_batch_device(n, m, k, ptr, vtx, dem) as h:
        h.kernelize()
        assert h.work_stats() == (0, 0)  # by candidate lists
        for b in range(0, len(order), 5):
            _same(h.result(b), refs[order[b]], b)
    for b in (1, 2, 9):  # (long rows in instances 1 and 2, 8 and 9)
        start = int(ptr[int(m[:b].sum())])
        bad = vtx.clone()
        bad[start + 3] = int(n[b])
        with pytest.raises(mhs.MhsError) as ei:
            mhs.Instance.load_batch_device(n, m, k, ptr, bad, dem)
        assert ei.value.status == mhs.MHS_EINVAL and f"instance {b} " in str(ei.value)


@pytest.mark.parametrize("n,m,lo,hi,fmin,fmax,leaves", [
    (2000, 4000, 24, 96, 1, 24, True), (1000, 1000, 150, 200, 1, 40, True),
    (1000, 4000, 150, 200, 1, 4, False), (300, 400, 20, 60, 1, 20, False),
    (4000, 8000, 2, 16, 100, 100, False), (1000, 20000, 8, 16, 1, 8, False)])
def test_large_demands_choose_the_path_that_pays(mhs, n, m, lo, hi, fmin, fmax, leaves):
    """Walks that find many pairs to be decided row by row count for more."""
    rng = np.random.Generator(np.random.PCG64(n + m + fmax))
    inst = I.from_edges(n, [np.sort(rng.choice(n, rng.integers(lo, hi + 1), replace=False)) for _ in range(m)],
                        rng.integers(fmin, fmax + 1, m), k=4)
    with mhs.Instance.load(inst) as h:
        h.kernelize()
        assert (h.work_stats()[1] > 0) == leaves
        got = h.result()
    _same(got, mhs.kernelize(inst, contraction="popcount"))


def test_one_hyperedge_of_a_large_demand_leaves_the_lists(mhs):
    rng = np.random.Generator(np.random.PCG64(600))
    rows = [np.sort(rng.choice(3000, 10, replace=False)) for _ in range(9000)] + [np.arange(600)]
    inst = I.from_edges(3000, rows, [2] * 9000 + [600], k=4)
    with mhs.Instance.load(inst) as h:
        h.kernelize()
        assert h.work_stats()[1] > 0
        got = h.result()
    _same(got, mhs.kernelize(inst, contraction="popcount"))


def _shared(kind, c, h, m, f, seed):
    """h long hyperedges over c common vertices beside m small ones."""
    rng = np.random.Generator(np.random.PCG64(seed))
    if kind == "twins":  # (and one vertex of its own each)
        rows = [np.append(np.arange(c), c + q) for q in range(h)]
    elif kind == "complement":  # every vertex misses one hyperedge
        h = c
        rows = [np.delete(np.arange(c), q) for q in range(h)]
    else:
        rows = [np.nonzero(rng.random(c) < 0.95)[0] for _ in range(h)]
    lo = c + h
    rows += [lo + np.sort(rng.choice(900, 6, replace=False)) for _ in range(m)]
    return I.from_edges(lo + 900, rows, [f] * h + [2] * m, k=3)


@pytest.mark.parametrize("kind,c,h,m,f", [
    ("twins", 400, 20, 900, 1), ("twins", 400, 20, 900, 7), ("twins", 300, 300, 900, 2),
    ("subsets", 300, 40, 900, 2), ("complement", 230, 230, 900, 1), ("complement", 60, 60, 0, 1),
    ("complement", 300, 300, 3000, 1), ("twins", 400, 20, 900, 100)])
def test_vertices_of_nearly_equal_hyperedges(mhs, kind, c, h, m, f):
    """MD tests that go far: many members, most of them in most hyperedges."""
    inst = _shared(kind, c, h, m, f, c + h)
    for fe in (False, True):
        ref = mhs.kernelize(inst, contraction="popcount", full_edges=fe)
        _same(mhs.kernelize(inst, full_edges=fe), ref)
        with mhs.Instance.load_batch([inst] * 180, full_edges=fe) as hd:
            hd.kernelize()
            _same(hd.result(0), ref)
            _same(hd.result(179), ref)


@pytest.mark.parametrize("n,m,share,leaves", [(60, 2000, .85, True), (250, 500, .9, True),
                                              (250, 500, .6, False), (30, 2000, .9, False)])
def test_dense_hypergraphs_go_to_the_contraction(mhs, n, m, share, leaves):
    rng = np.random.Generator(np.random.PCG64(n))
    inst = I.from_edges(n, [np.nonzero(rng.random(n) < share)[0] for _ in range(m)],
                        rng.integers(1, 3, m), k=4)
    ref = mhs.kernelize(inst, contraction="popcount")
    with mhs.Instance.load(inst) as h:
        h.kernelize()
        assert (h.work_stats()[1] > 0) == leaves
        _same(h.result(), ref)
    if inst.nnz <= 65536:
        _noalloc(mhs, inst, ref)


def test_server_budget_covers_the_lists(mhs):
    """What a group of requests holds by candidate lists is reserved too, and
    where the budget has no room for that, the device loop takes them."""
    inst = I.uniform_random(100, 200, 2, 8, 3, 5, seed=1)
    ref = O.reduce(inst)
    lists = 16 * 16384 + 8 * 65536  # tasks and pairs of a request alone, at least
    for budget in (0, 600 << 10):
        with mhs.Server(hbm_budget_bytes=budget) as srv:
            for _ in range(3):
                _same(srv.poll(srv.submit(inst)), ref, budget)
            st = srv.stats()
        assert st["completed"] == 3 and st["bytes_in_use"] == 0
        if budget:
            assert st["peak_bytes"] <= budget
        else:
            assert st["peak_bytes"] >= lists
    wide = I.uniform_random(256, 4000, 180, 200, 2, 5, seed=2)
    for budget in (8 << 20, 64 << 20):
        with mhs.Server(hbm_budget_bytes=budget) as srv:
            tickets = [srv.submit(i) for i in (wide, inst, inst, wide, inst)]
            for t, i in zip(tickets, (wide, inst, inst, wide, inst)):
                _same(srv.poll(t), ref if i is inst else mhs.kernelize(wide), budget)
            st = srv.stats()
        assert st["peak_bytes"] <= budget and st["bytes_in_use"] == 0


def test_server_group_that_fails_goes_to_the_device_loop(mhs):
    """An error of a group's launch is not every request's result."""
    insts = [I.uniform_random(n, 2 * n, 2, 8, 3, 5, seed=n) for n in (300, 900, 2000)]
    for fe in (False, True):
        refs = [O.reduce_variant(i, "dp", fe) for i in insts]
        mhs.selftest_team_wait(1_000_000)
        srv = mhs.Server(full_edges=fe)
        mhs.selftest_team_wait(0)
        try:
            for _ in range(2):
                tickets = [srv.submit(i) for i in insts]
                for t, ref in zip(tickets, refs):
                    got = srv.poll(t)
                    _same(got, ref)
                    if fe:
                        assert got["forced"].tolist() == ref["forced"].tolist()
        finally:
            srv.close()


@pytest.mark.parametrize("fe", [False, True])
def test_server_group_that_does_not_pay(mhs, fe):
    """Requests whose build says that the lists do not pay, alone and among
    others: all of the group take slots of the device loop."""
    rng = np.random.Generator(np.random.PCG64(55))
    wide = I.from_edges(300, [np.sort(rng.choice(300, rng.integers(20, 61), replace=False))
                              for _ in range(3000)], rng.integers(1, 21, 3000), k=4)
    with mhs.Instance.load(wide) as h:
        h.kernelize()
        assert h.work_stats()[1] > 0  # contracted
    insts = [wide, I.uniform_random(400, 900, 2, 8, 3, 5, seed=3), I.uniform_random(90, 200, 2, 5, 3, 5, seed=4)]
    refs = [mhs.kernelize(i, contraction="popcount", full_edges=fe) for i in insts]
    with mhs.Server(full_edges=fe) as srv:
        _same(srv.poll(srv.submit(wide)), refs[0])
        srv.pause(True)
        tickets = [srv.submit(i) for i in insts]
        srv.pause(False)
        for t, ref in zip(tickets, refs):
            _same(srv.poll(t), ref)


@pytest.mark.parametrize("rule,fe", VARIANTS)
def test_large_demands_where_the_lists_do_not_pay(mhs, rule, fe):
    """Demands that FP32 tests would round are decided in 32-bit integers by
    every entry point that chooses its form itself."""
    import torch
    rng = np.random.Generator(np.random.PCG64(23))
    insts = []
    for n, m, lo, hi in ((60, 300, 40, 60), (300, 3000, 20, 60), (700, 60, 300, 500), (200, 300, 2, 9)):
        rows = [np.sort(rng.choice(n, rng.integers(lo, hi + 1), replace=False)) for _ in range(m)]
        top = int(rng.choice([2**23, 2**25, 2**30, TOP - 40]))
        insts.append(I.from_edges(n, rows, top + rng.integers(0, 40, m), k=4))
        insts.append(I.from_edges(n, rows, rng.choice([1, 2, top, top + 3], m), k=4))
    opts = {"rule": rule, "full_edges": fe}
    refs = [O.reduce_variant(i, rule, fe) for i in insts]
    for b, (inst, ref) in enumerate(zip(insts, refs)):
        _same(mhs.kernelize(inst, **opts), ref, f"host {b}")
        d = _dev(inst.edge_ptr, inst.edge_vtx, inst.demand)
        with mhs.Instance.load_device(inst.n, inst.m, *d, inst.k, **opts) as h:
            h.kernelize()
            assert h.work_stats() == (0, 0)
            _same(h.result(), ref, f"device {b}")
        for part in ([inst], [inst, insts[-1]]):
            with mhs.Instance.load_batch(part, **opts) as h:
                h.kernelize()
                _same(h.result(0), ref, f"batch {b}")
            n, m = (np.array([getattr(i, x) for i in part], np.int32) for x in "nm")
            ptr = torch.from_numpy(np.concatenate(
                [[0], np.cumsum(np.concatenate([np.diff(i.edge_ptr) for i in part]))])).cuda()
            vtx, dem = _dev(np.concatenate([i.edge_vtx for i in part]),
                            np.concatenate([i.demand for i in part]))
            k = np.array([i.k for i in part], np.int64)
            with mhs.Instance.load_batch_device(n, m, k, ptr, vtx, dem, **opts) as h:
                h.kernelize()
                _same(h.result(0), ref, f"device batch {b}")
    small = I.uniform_random(400, 900, 2, 8, 3, 5, seed=3)
    sref = O.reduce_variant(small, rule, fe)
    with mhs.Server(**opts) as srv:
        srv.pause(True)
        tickets = [srv.submit(i) for i in insts + [small]]
        srv.pause(False)
        for b, (t, ref) in enumerate(zip(tickets, refs + [sref])):
            got = srv.poll(t)
            _same(got, ref, f"server {b}")
            if fe:
                assert got["forced"].tolist() == ref["forced"].tolist()
        st = srv.stats()
    assert st["completed"] == len(tickets) and st["active"] == 0 and st["bytes_in_use"] == 0


def test_no_memory_for_the_contraction():
    """A load whose lists do not pay stays on them where the operands of the
    contraction (9.8 GB here) find no memory.  (A process of its own, most of the
    card's memory taken; nothing cached by other tests.)"""
    import subprocess
    import sys
    code = """
import numpy as np, torch
from oracle import oracle as O
from paper_2109_06042_gb300 import instances as I, mhs
rng = np.random.Generator(np.random.PCG64(70))
n = m = 70000
rows = [np.unique(r) for r in rng.integers(0, n, (m, 3))] + [np.sort(rng.choice(n, 6000, replace=False))]
inst = I.from_edges(n, rows, np.append([min(2, len(r)) for r in rows[:-1]], 6000), k=3)
ref = O.reduce(inst)
d = [torch.from_numpy(np.ascontiguousarray(a, np.int32)).cuda() for a in (inst.edge_ptr, inst.edge_vtx, inst.demand)]
fill = torch.empty(torch.cuda.mem_get_info()[0] - (6 << 30), dtype=torch.uint8, device='cuda')
for load in (lambda: mhs.Instance.load(inst), lambda: mhs.Instance.load_device(n, inst.m, *d, inst.k),
             lambda: mhs.Instance.load_batch([inst])):
    with load() as h:
        h.kernelize()
        got = h.result()
    for key in ('vertices', 'edges', 'demands'):
        assert got[key].tolist() == ref[key].tolist(), key
    assert got['rounds'] == ref['rounds']
try:
    mhs.kernelize(inst, contraction='fp8')
    raise SystemExit('the contraction found memory')
except mhs.MhsError as e:
    assert e.status == mhs.MHS_ENOMEM
"""
    import os
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
