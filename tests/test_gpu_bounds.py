"""The vertex bounds that delete hyperedges before the FP8 operand is built,
against the oracle: equal hyperedges of one vertex (the lower index stays), a
vertex listed twice, bounds from one vertex and from several, both rules, FE
after it, instances alone (from 8,000 hyperedges on) and in a batch, and the
sizes recorded per round."""
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


def _singles(n, m, seed):
    """Mostly hyperedges of one or two vertices, demands up to 4."""
    rng = np.random.Generator(np.random.PCG64(seed))
    edges = [np.sort(rng.choice(n, rng.choice([1, 1, 2, 2, 3, 7], p=[.2, .2, .2, .2, .1, .1]),
                                replace=False)).tolist() for _ in range(m)]
    return I.from_edges(n, edges, rng.integers(1, 5, m), k=4)


CASES = [_singles(9, 5, 1), _singles(30, 31, 2), _singles(40, 257, 3), _singles(2000, 1025, 4),
         _singles(900, 2049, 5), _singles(3000, 8001, 6), _singles(9000, 8193, 7),
         I.config_powerlaw(6, n=4500, m=9000)]


def _rows(inst):
    return [inst.edge_vtx[a:b].tolist() for a, b in zip(inst.edge_ptr[:-1], inst.edge_ptr[1:])]


@pytest.mark.parametrize("rule,fe", VARIANTS)
def test_alone_and_in_a_batch(mhs, rule, fe):
    refs = [O.reduce_variant(i, rule, fe) for i in CASES]
    with mhs.Instance.load_batch(CASES, contraction="fp8", rule=rule, full_edges=fe) as h:
        h.kernelize()
        got = [h.result(b) for b in range(len(CASES))]
    got += [mhs.kernelize(i, contraction="fp8", rule=rule, full_edges=fe) for i in CASES]
    for g, ref in zip(got, refs + refs):
        for key in ("vertices", "edges", "demands"):
            assert g[key].tolist() == ref[key].tolist(), key
        assert g["k"] == ref["k"] and g["rounds"] == ref["rounds"]


@pytest.mark.parametrize("rule", ["dp", "se"])
def test_vertices_listed_twice(mhs, rule):
    import torch
    rng = np.random.Generator(np.random.PCG64(8))
    for inst in CASES:
        rows = [rng.permutation(r + r[:rng.integers(0, len(r) + 1)]) for r in _rows(inst)]
        ptr = np.concatenate([[0], np.cumsum([len(r) for r in rows])])
        d = [torch.from_numpy(np.ascontiguousarray(a, np.int32)).cuda()
             for a in (ptr, np.concatenate(rows), inst.demand)]
        ref = O.reduce_variant(inst, rule, False)
        with mhs.Instance.load_device(inst.n, inst.m, *d, inst.k, contraction="fp8", rule=rule) as h:
            h.kernelize()
            got = h.result()
        assert got["vertices"].tolist() == ref["vertices"].tolist()
        assert got["edges"].tolist() == ref["edges"].tolist() and got["rounds"] == ref["rounds"]


def test_sizes_per_round_equal_the_bit_packed_form(mhs):
    for inst in CASES:
        rec = []
        for form in ("fp8", "popcount"):
            with mhs.Instance.load(inst, contraction=form) as h:
                stats = []
                while not stats or stats[-1]["changed"]:
                    stats.append(h.reduce_round())
                rec.append((stats, h.trace()[0].tolist()))
        assert rec[0] == rec[1]


@pytest.mark.parametrize("count", [64, 65])
def test_operand_groups_of_8_and_of_32_rows(mhs, count):
    """Loads of up to and above 65,536 rows set the operand by 8 and by 32 rows
    a warp; rows of 30 to 40 vertices overflow the warp's table in both."""
    insts = [I.uniform_random(300, 1024, 1, 6, 3, 0, seed=1), I.uniform_random(300, 1024, 30, 40, 3, 0, seed=2),
             I.uniform_random(290, 1024, 1, 40, 3, 0, seed=3)]
    refs = [O.reduce(i) for i in insts]
    with mhs.Instance.load_batch([insts[b % 3] for b in range(count)], contraction="fp8") as h:
        h.kernelize()
        for b in range(count):
            got, ref = h.result(b), refs[b % 3]
            assert got["vertices"].tolist() == ref["vertices"].tolist(), b
            assert got["edges"].tolist() == ref["edges"].tolist() and got["rounds"] == ref["rounds"]
