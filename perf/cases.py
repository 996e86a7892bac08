"""The work users of this library have it do, as cases to be timed.

Every case is one whole kernelization through the public entry points:
loading the hypergraph, Algorithm 3 to its fixpoint, and the result.  Sizes
and distributions are those of the repository's generators
(``paper_2109_06042_gb300/instances.py``); they are drawn here with torch on
the GPU, so that large inputs are made quickly.

A case is a dict:

* ``family``       shape of the hypergraph: ``uniform`` (|e| uniform in
                   [smin, smax], distinct uniform vertices), ``powerlaw``
                   (P(|e| = s) ~ s^-2.5 on 2..64, Zipf(1.1) vertices),
                   ``interval`` (intervals on a line of mean length ``mean``,
                   5 % noise), ``batch`` (many uneven uniform instances) or
                   ``stream`` (requests to the server);
* ``n``, ``m``     vertices and hyperedges of a single instance; ``count``
                   instances of a batch, or requests;
* ``entry``        how the program calls: ``device`` (CSR in GPU memory,
                   masks to GPU memory), ``host`` (``mhs.kernelize`` on host
                   arrays), ``noalloc`` (``mhs.kernelize_noalloc``) or
                   ``server``;
* ``contraction``, ``rule``, ``full_edges``  the options of the same names.
"""
import numpy as np
import torch

from paper_2109_06042_gb300 import instances, mhs


def _single(name, family, n, m, smin=2, smax=16, alpha=3, mean=0, entry="device",
            contraction="auto", rule="dp", full_edges=False):
    return {"name": name, "family": family, "n": n, "m": m, "smin": smin, "smax": smax,
            "alpha": alpha, "mean": mean, "entry": entry, "contraction": contraction,
            "rule": rule, "full_edges": full_edges}


def _many(name, family, count, nmin, nmax, mfac, entry, rule="dp", full_edges=False):
    return {"name": name, "family": family, "count": count, "nmin": nmin, "nmax": nmax,
            "mfac": mfac, "smin": 2, "smax": 16, "alpha": 3, "entry": entry,
            "contraction": "auto", "rule": rule, "full_edges": full_edges}


def listed():
    return [
        # the smallest call: the plain single-instance workload, where latency counts
        _single("uniform_200x400", "uniform", 200, 400, smax=8),
        # a caller that may not allocate: small instance, caller's buffers
        _single("noalloc_1000x2000", "uniform", 1000, 2000, entry="noalloc"),
        # the one-line use from Python: host arrays in, ids out
        _single("host_1000x2000", "uniform", 1000, 2000, entry="host"),
        # the integer-unit form, chosen by a caller who wants no tensor cores
        _single("popcount_4000x8000", "uniform", 4000, 8000, contraction="popcount"),
        # large hyperedges: the densest hypergraphs
        _single("wide_2000x4000", "interval", 2000, 4000, smax=0, alpha=4, mean=64),
        # the largest requests of the serving stream, alone
        _single("uniform_16000x32000", "uniform", 16000, 32000),
        # the headline workload: skewed sizes and degrees
        _single("powerlaw_20000x40000", "powerlaw", 20000, 40000, smax=64, alpha=4),
        # the same with the tensor-core form asked for by name
        _single("powerlaw_fp8", "powerlaw", 20000, 40000, smax=64, alpha=4, contraction="fp8"),
        # the variant with the superedge rule and full edges, from host arrays
        _single("powerlaw_se_fe", "powerlaw", 20000, 40000, smax=64, alpha=4, entry="host",
                rule="se", full_edges=True),
        # low Dilworth number: the largest single instance
        _single("interval_50000x100000", "interval", 50000, 100000, smax=0, alpha=2,
                mean=12),
        # throughput over many independent uneven instances
        _many("batch_4096", "batch", 4096, 50, 2000, 2, "device"),
        # a burst of requests to a running server
        _many("server_128", "stream", 128, 100, 20000, 3, "server"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["uniform", "uniform", "noalloc", "host", "popcount", "wide", "powerlaw",
                       "interval", "batch", "server"])
    # the variants are options of every entry point but the allocation-free one
    rule = rng.choice(["dp", "dp", "dp", "se"])
    fe = rng.random() < 0.25
    if kind == "powerlaw":
        n = _log_uniform(rng, 1000, 20000)
        case = _single("", kind, n, rng.randint(n, 2 * n), smax=64, alpha=4,
                       entry=rng.choice(["device", "host"]),
                       contraction=rng.choice(["auto", "fp8"]), rule=rule, full_edges=fe)
    elif kind == "interval":
        n = _log_uniform(rng, 2000, 50000)
        case = _single("", kind, n, rng.randint(n, 2 * n), smax=0, alpha=2,
                       mean=rng.randint(6, 16), rule=rule, full_edges=fe)
    elif kind == "wide":
        n = _log_uniform(rng, 300, 2000)
        case = _single("", "interval", n, rng.randint(n, 2 * n), smax=0, alpha=4,
                       mean=rng.randint(24, 96), rule=rule, full_edges=fe)
    elif kind == "batch":
        case = _many("", kind, _log_uniform(rng, 8, 4096), 50, _log_uniform(rng, 200, 2000), 2,
                     "device", rule=rule, full_edges=fe)
    elif kind == "server":
        case = _many("", "stream", _log_uniform(rng, 4, 128), 100, _log_uniform(rng, 1000, 20000),
                     3, "server", rule=rule, full_edges=fe)
    elif kind == "popcount":
        n = _log_uniform(rng, 100, 4000)
        case = _single("", "uniform", n, rng.randint(n, 2 * n), contraction="popcount", rule=rule,
                       full_edges=fe)
    elif kind == "noalloc":
        n = _log_uniform(rng, 50, 2000)
        case = _single("", "uniform", n, rng.randint(n, 2 * n), entry="noalloc")
    else:
        n = _log_uniform(rng, 100, 16000 if kind == "uniform" else 4000)
        case = _single("", "uniform", n, rng.randint(n, 2 * n), smax=rng.choice([8, 16]),
                       entry="host" if kind == "host" else "device", rule=rule, full_edges=fe)
    del case["name"]
    return case


# ------------------------------------------------------------------ inputs --

def _gpu():
    return torch.device("cuda", torch.cuda.current_device())


def _distinct(sizes, draw_rows, g):
    """Row r: sizes[r] distinct ids, ascending, in a matrix padded with a
    large value.  draw_rows(rows, width) draws ids for the given rows; entries
    that repeat another entry of their row are drawn again."""
    dev = sizes.device
    width = int(sizes.max())
    pad = 1 << 40
    out = torch.empty((sizes.numel(), width), dtype=torch.int64, device=dev)
    rows = torch.arange(sizes.numel(), device=dev)
    valid = torch.arange(width, device=dev)[None, :] < sizes[:, None]
    cur = torch.where(valid, draw_rows(rows, width), pad)
    while True:
        cur = cur.sort(dim=1).values
        dup = torch.zeros_like(cur, dtype=torch.bool)
        dup[:, 1:] = (cur[:, 1:] == cur[:, :-1]) & (cur[:, 1:] < pad)
        bad = dup.any(dim=1)
        out[rows[~bad]] = cur[~bad]
        rows, cur, dup = rows[bad], cur[bad], dup[bad]
        if rows.numel() == 0:
            return out, valid
        cur = torch.where(dup, draw_rows(rows, width), cur)


def _demands(sizes, alpha, g):
    u = torch.rand(sizes.numel(), device=sizes.device, generator=g, dtype=torch.float64)
    hi = torch.clamp(sizes, max=alpha)
    return (1 + (u * hi).floor().clamp(max=hi - 1)).to(torch.int32)


def _uniform_rows(nrow, smin, smax, alpha, g):
    """Hyperedges with |e| ~ U{smin..smax} over the vertices 0 .. nrow[r] - 1."""
    sizes = torch.randint(smin, smax + 1, nrow.shape, device=nrow.device, generator=g)
    sizes = torch.minimum(sizes, nrow)

    def rows_of(rows, width):
        u = torch.rand((rows.numel(), width), device=nrow.device, generator=g,
                       dtype=torch.float64)
        hi = nrow[rows][:, None]
        return torch.minimum((u * hi).long(), hi - 1)

    mat, valid = _distinct(sizes, rows_of, g)
    return sizes, mat[valid].to(torch.int32), _demands(sizes, alpha, g)


def _powerlaw_rows(n, m, smax, alpha, g):
    dev = g.device
    s = torch.arange(2, smax + 1, device=dev, dtype=torch.float64)
    p = s ** -2.5
    sizes = 2 + torch.multinomial(p / p.sum(), m, replacement=True, generator=g)
    perm = torch.randperm(n, device=dev, generator=g)
    pop = (torch.arange(n, device=dev, dtype=torch.float64) + 1.0) ** -1.1
    cdf = torch.cumsum(pop, 0) / pop.sum()

    def rows_of(rows, width):
        u = torch.rand((rows.numel(), width), device=dev, generator=g, dtype=torch.float64)
        return perm[torch.searchsorted(cdf, u).clamp(max=n - 1)]

    mat, valid = _distinct(sizes, rows_of, g)
    return sizes, mat[valid].to(torch.int32), _demands(sizes, alpha, g)


def _interval_rows(n, m, mean, alpha, g):
    """Intervals with geometric lengths, 5 % of the members
    replaced by uniform vertices, then deduplicated."""
    dev = g.device
    start = torch.randint(0, n, (m,), device=dev, generator=g)
    u = torch.rand(m, device=dev, generator=g, dtype=torch.float64)
    length = 1 + torch.floor(torch.log1p(-u) / np.log1p(-1.0 / mean)).long()
    length = torch.minimum(length, n - start)
    width = int(length.max())
    col = torch.arange(width, device=dev)[None, :]
    noise = torch.rand((m, width), device=dev, generator=g) < 0.05
    repl = torch.randint(0, n, (m, width), device=dev, generator=g)
    mem = torch.where(noise, repl, start[:, None] + col)
    mem = torch.where(col < length[:, None], mem, 1 << 40).sort(dim=1).values
    valid = mem < (1 << 40)
    valid[:, 1:] &= mem[:, 1:] != mem[:, :-1]
    sizes = valid.sum(dim=1)
    return sizes, mem[valid].to(torch.int32), _demands(sizes, alpha, g)


def _offsets(sizes, dtype):
    ptr = torch.zeros(sizes.numel() + 1, dtype=dtype, device=sizes.device)
    torch.cumsum(sizes, 0, out=ptr[1:])
    return ptr


def _budget(n):
    return n // 10


def _single_csr(case, seed):
    """(edge_ptr int64, edge_vtx int32, demand int32) of a single instance, on the GPU."""
    g = torch.Generator(device=_gpu())
    g.manual_seed(seed)
    n, m = case["n"], case["m"]
    if case["family"] == "powerlaw":
        sizes, vtx, dem = _powerlaw_rows(n, m, case["smax"], case["alpha"], g)
    elif case["family"] == "interval":
        sizes, vtx, dem = _interval_rows(n, m, case["mean"], case["alpha"], g)
    else:
        nrow = torch.full((m,), n, dtype=torch.int64, device=_gpu())
        sizes, vtx, dem = _uniform_rows(nrow, case["smin"], case["smax"], case["alpha"], g)
    return _offsets(sizes, torch.int64), vtx, dem


def _many_csr(case, seed):
    """Sizes of the instances (host; they belong to the case) and their
    concatenated CSR (GPU)."""
    rng = np.random.Generator(np.random.PCG64(4000))
    count, lo, hi = case["count"], case["nmin"], case["nmax"]
    if case["family"] == "stream":  # log-uniform sizes
        n = np.rint(np.exp(rng.uniform(np.log(lo), np.log(hi), count))).astype(np.int64)
    else:
        n = rng.integers(lo, hi + 1, count)
    m = np.array([rng.integers(x, case["mfac"] * x + 1) for x in n], dtype=np.int64)
    g = torch.Generator(device=_gpu())
    g.manual_seed(seed)
    dev_n, dev_m = torch.from_numpy(n).to(_gpu()), torch.from_numpy(m).to(_gpu())
    nrow = torch.repeat_interleave(dev_n, dev_m)
    sizes, vtx, dem = _uniform_rows(nrow, case["smin"], case["smax"], case["alpha"], g)
    return n, m, _offsets(sizes, torch.int64), vtx, dem


def _host_instance(n, ptr, vtx, dem):
    return instances.Instance(n=int(n), m=len(dem), edge_ptr=ptr.astype(np.int32), edge_vtx=vtx,
                              demand=dem, k=_budget(int(n)))


def _split(case, seed):
    """The instances of a batch or stream as host arrays."""
    n, m, ptr, vtx, dem = _many_csr(case, seed)
    ptr, vtx, dem = ptr.cpu().numpy(), vtx.cpu().numpy(), dem.cpu().numpy()
    e = np.concatenate([[0], np.cumsum(m)])
    out = []
    for b in range(len(n)):
        p = ptr[e[b]:e[b + 1] + 1]
        out.append(_host_instance(n[b], p - p[0], vtx[p[0]:p[-1]].copy(), dem[e[b]:e[b + 1]].copy()))
    return out


def prepare(case, seed):
    opts = {"contraction": case["contraction"], "rule": case["rule"],
            "full_edges": case["full_edges"]}
    state = {"entry": case["entry"], "family": case["family"], "opts": opts}
    if case["entry"] == "server":
        state["requests"] = _split(case, seed)
        state["server"] = mhs.Server(**opts)
        return state
    if case["family"] == "batch":
        n, m, ptr, vtx, dem = _many_csr(case, seed)
        state.update(n=n.astype(np.int32), m=m.astype(np.int32), k=n // 10, ptr=ptr, vtx=vtx,
                     dem=dem)
        total_n, total_m = int(n.sum()), int(m.sum())
    else:
        ptr, vtx, dem = _single_csr(case, seed)
        if case["entry"] == "host":
            state["inst"] = _host_instance(case["n"], ptr.cpu().numpy(), vtx.cpu().numpy(),
                                           dem.cpu().numpy())
            return state
        state.update(n=case["n"], m=case["m"], k=_budget(case["n"]), ptr=ptr.to(torch.int32),
                     vtx=vtx, dem=dem)
        total_n, total_m = case["n"], case["m"]
    state["alive_v"] = torch.empty(total_n, dtype=torch.uint8, device=_gpu())
    state["alive_e"] = torch.empty(total_m, dtype=torch.uint8, device=_gpu())
    state["stream"] = torch.cuda.Stream()  # the library's work runs on it, as in bench.py
    torch.cuda.synchronize()
    return state


def _by_id(ids, values, size):
    """A value for every input id: the given ones at the ids, 0 elsewhere."""
    out = np.zeros(size, np.int32)
    out[ids] = values
    return out


def _answer(n, m, res):
    """mhs.kernelize's lists, spread over the input ids (the lists' lengths
    depend on the input)."""
    out = {"alive_v": _by_id(res["vertices"], 1, n), "demand": _by_id(res["edges"],
                                                                      res["demands"], m),
           "k": res["k"], "rounds": res["rounds"]}
    if "forced" in res:
        out["forced"] = _by_id(res["forced"], 1, n)
    return out


def run(state):
    opts = state["opts"]
    if state["entry"] == "server":
        srv = state["server"]
        tickets = [srv.submit(inst) for inst in state["requests"]]
        answers = [_answer(i.n, i.m, srv.poll(t)) for i, t in zip(state["requests"], tickets)]
        return {key: np.concatenate([np.atleast_1d(a[key]) for a in answers])
                for key in answers[0]}
    if state["entry"] == "host":
        inst = state["inst"]
        return _answer(inst.n, inst.m, mhs.kernelize(inst, **opts))
    av, ae = state["alive_v"], state["alive_e"]
    if state["entry"] == "noalloc":
        rounds = mhs.kernelize_noalloc(state["n"], state["m"], state["ptr"], state["vtx"],
                                       state["dem"], state["vtx"].numel(), av, ae,
                                       stream=state["stream"])
        return {"alive_v": av, "alive_e": ae, "rounds": rounds}
    if state["family"] == "batch":
        with mhs.Instance.load_batch_device(state["n"], state["m"], state["k"], state["ptr"],
                                            state["vtx"], state["dem"], stream=state["stream"],
                                            **opts) as h:
            stats = h.kernelize()
            h.result_batch_device(av, ae)
    else:
        with mhs.Instance.load_device(state["n"], state["m"], state["ptr"], state["vtx"],
                                      state["dem"], state["k"], stream=state["stream"],
                                      **opts) as h:
            stats = h.kernelize()
            h.result_device(av, ae)
    return {"alive_v": av, "alive_e": ae, "rounds": stats["rounds"],
            "n_alive": stats["n_alive"], "m_alive": stats["m_alive"]}


def work(case):
    """The hypergraph read once and the result written once.  The rules test
    sets of integers: no floating-point operation has to be done."""
    if case["family"] in ("batch", "stream"):
        lo, hi = case["nmin"], case["nmax"]
        mean_n = (hi - lo) / np.log(hi / lo) if case["family"] == "stream" else (lo + hi) / 2
        n = case["count"] * mean_n
        m = n * (1 + case["mfac"]) / 2
        size = (case["smin"] + case["smax"]) / 2
    else:
        n, m = case["n"], case["m"]
        if case["family"] == "powerlaw":
            s = np.arange(2, case["smax"] + 1, dtype=np.float64)
            size = float((s ** -1.5).sum() / (s ** -2.5).sum())
        elif case["family"] == "interval":
            size = float(case["mean"])
        else:
            size = (case["smin"] + case["smax"]) / 2
    return {"bytes": float(m * (4 * size + 8) + n + m), "flops": 0.0}


# ------------------------------------------------------------------- exact --

def _reduce64(n, ptr, vtx, dem, rule, full_edges):
    """Algorithm 3 (and rule FE at its fixpoints) in its matrix form, in 64
    bits: alive masks, demands, forced vertices and rounds."""
    dev = _gpu()
    ptr, vtx = ptr.to(dev).long(), vtx.to(dev).long()
    f = dem.to(dev).double().clone()
    m = f.numel()
    A = torch.zeros((m, n), dtype=torch.float64, device=dev)
    A[torch.repeat_interleave(torch.arange(m, device=dev), ptr[1:] - ptr[:-1]), vtx] = 1.0
    E, V = torch.arange(m, device=dev), torch.arange(n, device=dev)
    forced, rounds = [], 0
    while True:
        while True:
            rounds += 1
            before = E.numel() + V.numel()
            B = A[E][:, V]
            inter, size, fe = B @ B.T, B.sum(1), f[E]
            if rule == "se":
                D = (inter == size[:, None]) & (fe[:, None] >= fe[None, :])
            else:
                D = fe[:, None] - (size[:, None] - inter) >= fe[None, :]
            D.fill_diagonal_(False)
            first = torch.ones_like(D).triu(1)
            E = E[~(D & (~D.T | first)).any(0)]
            B = A[E][:, V]
            inter, deg = B.T @ B, B.sum(0)
            first = torch.ones((V.numel(), V.numel()), dtype=torch.bool, device=dev).triu(1)
            D = (inter == deg[None, :]) & ((inter != deg[:, None]) | first)
            D.fill_diagonal_(False)
            maxf = (B * f[E][:, None]).amax(0) if E.numel() else torch.zeros_like(deg)
            V = V[D.sum(0) < maxf]
            if E.numel() + V.numel() == before:
                break
        if not full_edges:
            break
        B = A[E][:, V]
        full = B.sum(1) == f[E]
        took = B[full].sum(0) > 0
        if not bool(full.any()):
            break
        f[E] -= B[:, took].sum(1)
        E = E[~full & (f[E] > 0)]
        forced.append(V[took])
        V = V[~took]
    forced = torch.cat(forced).sort().values if forced else torch.zeros(0, dtype=torch.int64)
    return V.cpu(), E.cpu(), f.cpu(), forced.cpu(), rounds


_EXACT_COST = 3e11  # m (m n) products of one round beyond which the 64-bit form takes too long


def _exact_ids(n, ptr, vtx, dem, case):
    if float(len(dem)) * len(dem) * n > _EXACT_COST:
        return None
    V, E, f, forced, rounds = _reduce64(n, ptr, vtx, dem, case["rule"], case["full_edges"])
    out = {"vertices": V.numpy(), "edges": E.numpy(), "demands": f[E].numpy(),
           "k": _budget(n) - forced.numel(), "rounds": rounds}
    if case["full_edges"]:
        out["forced"] = forced.numpy()
    return out


def exact(case, seed):
    if case["family"] in ("batch", "stream"):
        return None  # (many instances: too long in 64 bits)
    ptr, vtx, dem = _single_csr(case, seed)
    ids = _exact_ids(case["n"], ptr, vtx, dem, case)
    if ids is None:
        return None
    n, m = case["n"], case["m"]
    if case["entry"] == "host":
        return _answer(n, m, ids)
    out = {"alive_v": _by_id(ids["vertices"], 1, n), "alive_e": _by_id(ids["edges"], 1, m),
           "rounds": ids["rounds"]}
    if case["entry"] != "noalloc":
        out.update(n_alive=len(ids["vertices"]), m_alive=len(ids["edges"]))
    return out
