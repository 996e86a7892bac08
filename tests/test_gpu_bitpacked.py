"""The bit-packed passes (contraction="popcount") against the oracle, at the
edges of their blocks: 16 rows, 128 words (4,096 rows) of a bitmap, 512
members of a row gathered at a time, demands counted in unary (up to 4) and
in binary (above), repeated ids, equal hyperedges and both rules."""
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


def _nested(n, m, size, fmax, seed):
    """Rows of about `size` vertices that differ in a few, some of them equal."""
    rng = np.random.Generator(np.random.PCG64(seed))
    base = rng.permutation(n)[:size]
    edges = []
    for _ in range(m):
        drop = rng.integers(0, min(8, size))
        extra = rng.integers(0, n, rng.integers(0, 4))
        edges.append(sorted(set(base[drop:].tolist()) | set(extra.tolist())))
    return I.from_edges(n, edges, [int(rng.integers(1, fmax + 1)) for _ in edges], k=5)


CASES = [
    ("m15", I.uniform_random(40, 15, 1, 6, 3, 5, seed=1)),
    ("m17", I.uniform_random(33, 17, 1, 6, 5, 5, seed=2)),
    ("m4095", I.uniform_random(900, 4095, 1, 5, 4, 5, seed=3)),
    ("m4097", I.uniform_random(900, 4097, 1, 5, 6, 5, seed=4)),
    ("n4097", I.uniform_random(4097, 3000, 1, 12, 3, 5, seed=5)),
    ("n9000", I.uniform_random(9000, 8200, 2, 6, 4, 5, seed=6)),
    ("size511", _nested(700, 60, 511, 3, 7)),
    ("size513", _nested(2000, 60, 513, 4, 8)),
    ("size1500_f40", _nested(1600, 200, 1500, 40, 9)),
    ("size30_f4", _nested(64, 300, 30, 4, 10)),
    ("size30_f5", _nested(64, 300, 30, 5, 11)),
    ("size6_f9", _nested(12, 400, 6, 9, 12)),
]


@pytest.mark.parametrize("rule,fe", [("dp", False), ("se", False), ("dp", True), ("se", True)])
@pytest.mark.parametrize("name", [c[0] for c in CASES])
def test_equals_oracle(mhs, name, rule, fe):
    inst = dict(CASES)[name]
    ref = O.reduce_variant(inst, rule, fe)
    got = mhs.kernelize(inst, contraction="popcount", rule=rule, full_edges=fe)
    for key in ("vertices", "edges", "demands"):
        assert got[key].tolist() == ref[key].tolist(), key
    assert got["k"] == ref["k"] and got["rounds"] == ref["rounds"]


def test_repeated_ids_from_the_device(mhs):
    import torch
    inst = I.uniform_random(500, 1200, 1, 6, 5, 5, seed=13)
    rng = np.random.Generator(np.random.PCG64(14))
    rows = [rng.permutation(e + e[:rng.integers(0, len(e) + 1)]) for e in inst.edges()]
    ptr = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int32)
    d = [torch.from_numpy(np.ascontiguousarray(a, np.int32)).cuda()
         for a in (ptr, np.concatenate(rows), inst.demand)]
    ref = O.reduce(inst)
    with mhs.Instance.load_device(inst.n, inst.m, *d, inst.k, contraction="popcount") as h:
        h.kernelize()
        got = h.result()
    assert got["vertices"].tolist() == ref["vertices"].tolist()
    assert got["edges"].tolist() == ref["edges"].tolist() and got["rounds"] == ref["rounds"]


@pytest.mark.parametrize("n", [1, 31, 126, 127, 128, 254, 255, 256, 1023, 1024, 2047, 2048, 4095, 4096, 4098])
def test_vertices_in_all_hyperedges(mhs, n):
    """MD passes that walk whole lists: bitmaps of 1, 2, 4 .. 32 quads of words
    (a hyperedge per 1 .. 32 lanes) and more, lists of more than 512."""
    rng = np.random.Generator(np.random.PCG64(n))
    rows = [np.append(np.sort(rng.choice(n, min(n, 6), replace=False)), [n, n + 1]) for _ in range(1500)]
    inst = I.from_edges(n + 2, rows, np.full(1500, 3), k=5)
    ref = O.reduce(inst)
    got = mhs.kernelize(inst, contraction="popcount")
    for key in ("vertices", "edges", "demands"):
        assert got[key].tolist() == ref[key].tolist(), key
    assert got["rounds"] == ref["rounds"]
