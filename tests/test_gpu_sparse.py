"""The candidate-list path (what contraction="auto" takes for sparse
hypergraphs) against the oracle and the FP8 contraction, bit-exact: at the
edges of its lane groups (8), CTAs and teams, with long vertex lists (walked
as tasks, handled by whole CTAs), repeated and unsorted ids, demands above
the hyperedge's size, empty hyperedges, both rules, rule FE, single rounds,
sharded passes and batches, and on both sides of the rule that leaves it."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2109_06042_gb300 import instances as I

pytestmark = pytest.mark.gpu

VARIANTS = [("dp", False), ("se", False), ("dp", True), ("se", True)]


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
    if "forced" in got:
        assert got["forced"].tolist() == ref["forced"].tolist(), ctx


def _star(hubs, leaves, seed, alpha=2):
    """A few vertices in most hyperedges: lists far longer than a lane group's."""
    rng = np.random.Generator(np.random.PCG64(seed))
    edges = [sorted(set(rng.choice(hubs, rng.integers(0, 3)).tolist() +
                        (hubs + rng.choice(leaves, rng.integers(1, 4))).tolist()))
             for _ in range(4 * leaves)]
    return I.from_edges(hubs + leaves, edges,
                        [int(rng.integers(1, min(alpha, len(e)) + 1)) for e in edges], k=9)


def _cases():
    out = [I.uniform_random(n, m, lo, hi, a, 5, seed=n + m, name=f"u{n}x{m}_{lo}_{hi}")
           for n, m, lo, hi, a in [(7, 9, 1, 7, 3), (33, 31, 1, 8, 9), (64, 65, 7, 9, 4),
                                   (200, 400, 2, 8, 3), (513, 1025, 2, 17, 3), (1500, 2999, 1, 16, 4),
                                   (6000, 9001, 1, 6, 3)]]
    out += [I.from_edges(0, [], []), I.from_edges(5, [], []), I.from_edges(3, [[0, 1, 2]], [2]),
            _star(3, 40, 1), _star(2, 700, 2, alpha=4), _star(8, 1500, 3, alpha=3),
            I.config_interval(3, n=3000, m=6000), I.config_powerlaw(5, n=4000, m=8000)]
    return out


@pytest.mark.parametrize("rule,fe", VARIANTS)
def test_equals_oracle_and_contraction(mhs, rule, fe):
    for inst in _cases():
        ref = O.reduce_variant(inst, rule, fe)
        _same(mhs.kernelize(inst, rule=rule, full_edges=fe), ref, inst.name)
        _same(mhs.kernelize(inst, contraction="fp8", rule=rule, full_edges=fe), ref, inst.name)


@pytest.mark.parametrize("rule,fe", VARIANTS)
def test_tiny_with_loose_and_empty_hyperedges(mhs, rule, fe):
    insts = [I.tiny_random(s, nmax=24 if s % 2 else 16, mmax=24 if s % 3 else 12) for s in range(400)]
    rng = np.random.Generator(np.random.PCG64(77))
    for i in insts[::4]:  # demands far above the sizes
        i.demand[:] += rng.integers(0, 4, i.m).astype(np.int32)
    for s in range(40):  # empty hyperedges, several of equal demand
        e = I.tiny_random(1000 + s).edges() + [[], [], []]
        insts.append(I.from_edges(16, e, rng.integers(1, 4, len(e)), k=3))
    refs = [O.reduce_variant(i, rule, fe) for i in insts]
    with mhs.Instance.load_batch(insts, rule=rule, full_edges=fe) as h:
        h.kernelize()
        for b, (inst, ref) in enumerate(zip(insts, refs)):
            _same(h.result(b), ref, f"batch {b}")
    for b in range(0, len(insts), 7):
        _same(mhs.kernelize(insts[b], rule=rule, full_edges=fe), refs[b], f"alone {b}")


def test_device_rows_unsorted_and_with_repeats(mhs):
    import torch
    rng = np.random.Generator(np.random.PCG64(5))
    base = I.uniform_random(300, 500, 1, 20, 3, 5, seed=8)
    rows = []
    for e in base.edges():
        e = e + rng.choice(e, rng.integers(0, 3)).tolist()
        rng.shuffle(e)
        rows.append(e)
    ptr = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int32)
    vtx = np.concatenate(rows).astype(np.int32)
    dev = [torch.from_numpy(a).cuda() for a in (ptr, vtx, base.demand)]
    with mhs.Instance.load_device(base.n, base.m, *dev, base.k) as h:
        h.kernelize()
        _same(h.result(), O.reduce(base))


@pytest.mark.parametrize("what", ["ptr", "vertex", "demand"])
def test_malformed_device_inputs(mhs, what):
    import torch
    base = I.uniform_random(300, 500, 1, 20, 3, 5, seed=8)
    ptr, vtx, dem = base.edge_ptr.copy(), base.edge_vtx.copy(), base.demand.copy()
    if what == "ptr":
        ptr[100] = ptr[101] + 1
    elif what == "vertex":
        vtx[-1] = base.n
    else:
        dem[7] = 0
    dev = [torch.from_numpy(a).cuda() for a in (ptr, vtx, dem)]
    with pytest.raises(mhs.MhsError) as ei:
        mhs.Instance.load_device(base.n, base.m, *dev, base.k)
    assert ei.value.status == mhs.MHS_EINVAL


@pytest.mark.parametrize("fe", [False, True])
def test_rounds_one_by_one_trace_and_export(mhs, fe):
    inst = I.config_powerlaw(2, n=3000, m=6000)
    with mhs.Instance.load(inst, contraction="fp8", full_edges=fe) as ref, \
            mhs.Instance.load(inst, full_edges=fe) as h:
        while True:
            a, b = ref.reduce_round(), h.reduce_round()
            assert {k: a[k] for k in ("n_alive", "m_alive", "rounds", "changed", "active")} == \
                {k: b[k] for k in ("n_alive", "m_alive", "rounds", "changed", "active")}
            _same(h.result(), ref.result())
            if not a["active"]:
                break
        assert ref.trace()[0].tolist() == h.trace()[0].tolist()
        for x, y in zip(ref.export(), h.export()):
            assert np.array_equal(x, y)
    with mhs.Instance.load(inst, max_rounds=2) as h:
        assert h.kernelize()["rounds"] == 2
        _same(h.result(), O.reduce(inst, max_rounds=2))


@pytest.mark.parametrize("rule,fe", VARIANTS)
def test_sharded_passes(mhs, rule, fe):
    import torch
    inst = I.config_powerlaw(4, n=1500, m=3000)
    ref = O.reduce_variant(inst, rule, fe)
    hs = [mhs.Instance.load(inst, rule=rule, full_edges=fe) for _ in range(3)]
    while True:
        for phase in (0, 1):
            parts = []
            for r, h in enumerate(hs):
                h.pass_begin(phase)
                h.pass_contract(phase, r, 3)
                buf = torch.zeros(h.pass_elems(phase), device="cuda",
                                  dtype=torch.uint8 if phase == 0 else torch.int32)
                h.pass_partial(phase, buf)
                parts.append(buf)
            both = torch.stack(parts).amax(0) if phase == 0 else torch.stack(parts).sum(0).int()
            torch.cuda.synchronize()
            for h in hs:
                h.pass_merge(phase, both)
                st = h.pass_end(phase)
        if not st["active"]:
            break
    for h in hs:
        _same(h.result(), ref)
        h.free()


def test_batch_of_uneven_instances(mhs):
    insts = [I.config_batch_one(7000 + s) for s in range(40)] + \
        [I.from_edges(0, [], []), _star(4, 300, 9), I.config_uniform(3)]
    refs = [O.reduce(i) for i in insts]
    for part in (insts, insts[:5], insts[:2]):  # one CTA each; teams of CTAs
        with mhs.Instance.load_batch(part) as h:
            h.kernelize()
            for b in range(len(part)):
                _same(h.result(b), refs[b], f"{len(part)}: {b}")


@pytest.mark.parametrize("n", [3071, 3072, 3073])
def test_batch_around_the_limit_of_shared_vertices(mhs, n):
    """The build of a batch keeps the degrees and places of at most 3,072
    vertices in shared memory, and one CTA takes instances of both kinds in turn."""
    insts = [I.uniform_random(n + (s % 3 - 1) * 2, 3000 + s, 1, 6, 3, 5, seed=s) for s in range(3)]
    refs = [O.reduce(i) for i in insts]
    batch = [insts[b % 3] for b in range(700)]
    with mhs.Instance.load_batch(batch) as h:
        h.kernelize()
        for b in range(0, 700, 7):
            _same(h.result(b), refs[b % 3], f"{n}: {b}")


@pytest.mark.parametrize("size", [16, 17, 63, 64, 65, 96, 97, 700])
def test_rows_around_the_widths_of_the_build(mhs, size):
    """Rows of about `size` vertices of very uneven degrees, in order and not,
    with repeats (a group's registers, a warp's, the counting sort)."""
    import torch
    rng = np.random.Generator(np.random.PCG64(size))
    n, rows = 900, []
    weight = 1.0 / np.arange(1, n + 1) ** 1.2
    for i in range(300):
        r = rng.choice(n, size + int(rng.integers(-1, 2)), replace=False, p=weight / weight.sum())
        rows.append(r if i % 3 else np.concatenate([r, r[:rng.integers(0, 3)]]))
    rows = [np.sort(r) if i % 2 else r for i, r in enumerate(rows)] + rows[:5] + [r[1:] for r in rows[:9]]
    inst = I.from_edges(n, [sorted(set(r.tolist())) for r in rows], rng.integers(1, 5, len(rows)), k=2)
    ptr = np.concatenate([[0], np.cumsum([len(r) for r in rows])])
    d = [torch.from_numpy(np.ascontiguousarray(x, np.int32)).cuda()
         for x in (ptr, np.concatenate(rows), inst.demand)]
    ref = O.reduce(inst)
    with mhs.Instance.load_device(inst.n, inst.m, *d, inst.k) as h:
        h.kernelize()
        _same(h.result(), ref)
    _same(mhs.kernelize(inst), ref)


@pytest.mark.parametrize("rule", ["dp", "se"])
@pytest.mark.parametrize("deg", [31, 33, 47, 48, 49, 128, 129, 191, 193, 256, 257])
def test_lists_around_the_lengths_of_tasks(mhs, deg, rule):
    """Lists of `deg` hyperedges, alone among short ones and as the mean
    length; several rounds, with hyperedges of one vertex (bounds)."""
    rng = np.random.Generator(np.random.PCG64(deg))
    hubs = 6
    edges = [sorted({h, hubs + int(x), hubs + int(y)}) for h in range(hubs)
             for x, y in rng.integers(0, 90, (deg, 2))]
    edges += [[hubs + i] for i in range(0, 90, 7)]
    dense = [np.sort(rng.choice(40, 8, replace=False)).tolist() for _ in range(deg * 5)]
    for n, e in ((hubs + 90, edges), (40, dense)):
        inst = I.from_edges(n, e, rng.integers(1, 4, len(e)), k=3)
        _same(mhs.kernelize(inst, rule=rule), O.reduce_variant(inst, rule, False))


@pytest.mark.parametrize("n,m,lo,hi,alpha", [
    (1000, 2000, 2, 16, 3), (32, 4096, 14, 16, 3), (16, 4096, 16, 16, 3), (8, 4096, 1, 8, 5),
    (40, 4096, 14, 16, 8),
    (300, 300, 195, 205, 4), (1000, 60, 900, 1000, 9), (4096, 4096, 1, 16, 3)])
def test_noalloc_by_lists_and_by_bits(mhs, n, m, lo, hi, alpha):
    """mhs_kernelize_noalloc on both sides of the rule between its two forms."""
    import torch
    inst = I.uniform_random(n, m, lo, hi, alpha, 0, seed=n + m + lo)
    d = [torch.from_numpy(np.ascontiguousarray(a, np.int32)).cuda()
         for a in (inst.edge_ptr, inst.edge_vtx, inst.demand)]
    ref = O.reduce(inst)
    for _ in range(2):
        av = torch.full((n,), 7, dtype=torch.uint8, device="cuda")
        ae = torch.full((m,), 7, dtype=torch.uint8, device="cuda")
        rounds = mhs.kernelize_noalloc(n, m, *d, inst.nnz, av, ae)
        assert rounds == ref["rounds"]
        assert torch.nonzero(av).flatten().tolist() == ref["vertices"].tolist()
        assert torch.nonzero(ae).flatten().tolist() == ref["edges"].tolist()
        assert int(av.max()) <= 1 and int(ae.max()) <= 1


def test_dense_hypergraphs_are_contracted(mhs):
    """Long lists throughout: the load leaves this path, with the same result."""
    rng = np.random.Generator(np.random.PCG64(3))
    n, m = 2000, 20000
    sizes = rng.integers(300, 400, m)
    edges = [np.sort(rng.choice(n, s, replace=False)) for s in sizes]
    edges[5] = edges[4][:-2]
    inst = I.from_edges(n, edges, np.full(m, 2), k=5)
    inst.demand[5] = 3
    with mhs.Instance.load(inst) as h:
        h.kernelize()
        kb, _ = h.work_stats()
        assert kb > 0  # tensor-core work: the contraction ran
        got = h.result()
    _same(got, mhs.kernelize(inst, contraction="fp8"))


def test_threads_on_streams_of_their_own(mhs):
    """Teams of CTAs that wait on one another, from several threads at once."""
    import threading
    insts = [I.config_powerlaw(20 + s, n=4000, m=8000) for s in range(4)]
    refs = [O.reduce(i) for i in insts]
    errors = []

    def work(s):
        try:
            for _ in range(15):
                _same(mhs.kernelize(insts[s]), refs[s], f"thread {s}")
        except Exception as e:  # noqa: BLE001 (reported by the main thread)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(s,)) for s in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]
