"""Sharded rounds (mhs_pass_*) and mhs_kernelize on one handle, in turn."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2109_06042_gb300 import instances as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mhs():
    from paper_2109_06042_gb300 import build
    build.build()
    from paper_2109_06042_gb300 import mhs as M
    return M


def _fixpoint(n, m):
    """A large instance that the rules leave as it is, with full hyperedges."""
    inst = I.uniform_random(n, m, 3, 8, 4, 5, seed=1)
    res = O.reduce(inst)
    new = np.full(inst.n, -1)
    new[res["vertices"]] = np.arange(len(res["vertices"]))
    rows = inst.edges()
    edges = [[int(x) for x in new[rows[e]] if x >= 0] for e in res["edges"]]
    return I.from_edges(len(res["vertices"]), edges, res["demands"], k=5)


@pytest.mark.parametrize("contraction", ["fp8", "popcount", "auto"])
@pytest.mark.parametrize("rounds", [1, 2])
def test_kernelize_after_sharded_rounds(mhs, contraction, rounds):
    """The first round deletes nothing and rule FE fires; what the passes
    left behind (largest demands per vertex) is not taken for bounds."""
    inst = _fixpoint(12000, 12000)
    assert inst.m >= 8000 and any(len(e) == f for e, f in zip(inst.edges(), inst.demand))
    ref = O.reduce_variant(inst, "dp", True)
    with mhs.Instance.load(inst, contraction=contraction, full_edges=True) as h:
        for r in range(rounds):
            for phase in (0, 1):
                h.pass_begin(phase)
                h.pass_contract(phase, 0, 1)
                st = h.pass_end(phase)
            if r == 0:
                assert st["dp_deleted"] == st["md_deleted"] == 0 and st["active"]
        h.kernelize()
        got = h.result()
        for key in ("vertices", "edges", "demands"):
            assert got[key].tolist() == ref[key].tolist(), key
        assert got["k"] == ref["k"] and got["rounds"] == ref["rounds"]
        assert h.forced()[0].tolist() == ref["forced"].tolist()


@pytest.mark.parametrize("long", [64, 65, 900])
@pytest.mark.parametrize("rule", ["dp", "se"])
def test_vertex_bounds_leave_long_rows_to_the_contraction(mhs, rule, long):
    """Rows above 64 ids set no bounds and are not tested against them."""
    rng = np.random.Generator(np.random.PCG64(long))
    rows = [np.sort(rng.choice(2000, rng.integers(1, 6), replace=False)) for _ in range(8200)]
    rows += [np.sort(rng.choice(2000, long, replace=False)) for _ in range(30)]
    inst = I.from_edges(2000, rows, rng.integers(1, 5, len(rows)), k=3)
    inst.demand[8200:8215] = long
    ref = O.reduce_variant(inst, rule, False)
    got = mhs.kernelize(inst, contraction="fp8", rule=rule)
    for key in ("vertices", "edges", "demands"):
        assert got[key].tolist() == ref[key].tolist(), key
    assert got["rounds"] == ref["rounds"]


@pytest.mark.parametrize("contraction", ["fp8", "popcount", "auto"])
@pytest.mark.parametrize("rule", ["dp", "se"])
def test_full_edges_with_vertices_listed_twice(mhs, contraction, rule):
    """Device rows with repeats: a vertex counts once for a hyperedge's size and
    for the demand that it loses."""
    import torch
    rng = np.random.Generator(np.random.PCG64(16))
    for n, m, top in ((30, 40, 6), (60, 12, 50), (400, 900, 8), (252, 1, 214), (90, 300, 70)):
        rows = [rng.choice(n, rng.integers(1, top + 1), replace=False) for _ in range(m)]
        dem = [max(1, len(r) - int(rng.integers(0, 3))) for r in rows]
        inst = I.from_edges(n, [sorted(r.tolist()) for r in rows], dem, k=9)
        ref = O.reduce_variant(inst, rule, True)
        rep = [rng.permutation(np.concatenate([r, r[:rng.integers(0, len(r) + 1)], r[:1]])) for r in rows]
        d = [torch.from_numpy(np.ascontiguousarray(x, np.int32)).cuda()
             for x in (np.concatenate([[0], np.cumsum([len(r) for r in rep])]), np.concatenate(rep), inst.demand)]
        with mhs.Instance.load_device(n, m, *d, 9, contraction=contraction, rule=rule, full_edges=True) as h:
            h.kernelize()
            got = h.result()
            assert h.forced()[0].tolist() == ref["forced"].tolist()
        for key in ("vertices", "edges", "demands"):
            assert got[key].tolist() == ref[key].tolist(), (key, n, m)
        assert got["k"] == ref["k"] and got["rounds"] == ref["rounds"]
