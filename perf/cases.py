"""Performance cases: what a program built on this framework spends its GPU time on.

Nine kinds of work, each through the public entry points (``engine``, ``capacity`` and the C ABI of ``include/abm.h``):

  world      a predation world advanced by some steps (Section 5.1 of the paper), from a checkpoint or running on
  selective  the fused remove / distinct update / add call on a slab
  tick       one tick of a hand-written model on a slab: select, distinct update, remove, add
  sort       agents get new keys and live flags, then the slab is sorted by the key
  resolve    claims on resources, one winner each
  match      one matching round of many order books
  market     a session of order placement and matching, replayed from a CUDA graph
  batch      an ensemble of predation models advanced by some steps
  capacity   one epoch of training the capacity predictor, then its predictions

A case's fields say its sizes and options; ``draw`` spreads them over the range that real programs use.
"""
import math

import numpy as np
import torch

import workloads
from paper_2508_16508_gb300 import abm, capacity, engine


def listed():
    return [
        # the 40 x 40 world of the demonstrations and of interactive use: 200 steps from a saved start, launch latency
        dict(name="world_small", kind="world", side=40, sheep=100, wolves=25, cap_sheep=2048, cap_wolves=1024, warm=0,
             steps=200, resume=True, variant=0),
        # an ordinary study world on an odd lattice: resume from a checkpoint, run a stretch, write the next one
        dict(name="world_ordinary", kind="world", side=301, sheep=21600, wolves=5400, cap_sheep=180000,
             cap_wolves=90000, warm=40, steps=50, resume=True, variant=0),
        # the large world (2048 x 2048, 1M sheep, 250k wolves), a running simulation past its first transients
        dict(name="world_large", kind="world", side=2048, sheep=1_000_000, wolves=250_000, cap_sheep=8 << 20,
             cap_wolves=4 << 20, warm=300, steps=20, resume=False, variant=0),
        # the selective update at 2^24 slots x 8 fields, as in the benchmark: some, and half, of the agents touched
        dict(name="selective_some", kind="selective", n=1 << 24, fields=8, p=0.05),
        dict(name="selective_half", kind="selective", n=1 << 24, fields=8, p=0.5),
        # a model's own tick through the single calls, on an ordinary, ragged agent set
        dict(name="tick", kind="tick", n=100_003, fields=5, p=0.05, mask=False),
        # re-sorting agents by their cell after they moved (cells of a 2048 x 2048 lattice)
        dict(name="sort_by_cell", kind="sort", n=4_000_037, fields=8, bits=22, signed=False, live=0.5),
        # conflict resolution at the selective benchmark's scale, with its popular and unpopular resources
        dict(name="resolve", kind="resolve", claims=1 << 22, resources=1 << 18, zipf=1.1),
        # one matching round of 65,536 books of 1024 slots, half full
        dict(name="match", kind="match", books=65536, cap=1024, fill=0.5, spread=10),
        # the finance model's scale: 500 books of at most 1000 orders, 100 steps of placement and matching
        dict(name="market", kind="market", books=500, cap=1000, fill=0.2, traders=10, steps=100),
        # the ensemble of 4096 models of 16 to 256 cells a side at the paper's static shapes
        dict(name="batch", kind="batch", models=4096, side_lo=16, side_hi=256, steps=10, warm=60, extent=False),
        # training the capacity predictor: an epoch of batches of 1024 over 16384 trajectories, then all predictions
        dict(name="capacity_epoch", kind="capacity", rows=16384, rows_per_step=1024, hidden=128, layers=3),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["world", "world", "selective", "selective", "tick", "sort", "resolve", "match", "market", "batch",
                       "capacity"])
    if kind == "world":
        side = _log(rng, 24, 2048)
        cells = side * side
        sheep = max(8, int(cells * rng.uniform(0.05, 0.3)))
        wolves = max(2, int(sheep * rng.uniform(0.1, 0.4)))
        return dict(kind=kind, side=side, sheep=sheep, wolves=wolves, cap_sheep=2 * cells + 1000,
                    cap_wolves=cells + 1000, warm=rng.randint(0, 60), steps=_log(rng, 1, 20 if side > 600 else 100),
                    resume=side < 1024, variant=rng.choice([0, 0, 0, 1, 2, 3]))
    if kind == "selective":
        return dict(kind=kind, n=_log(rng, 10_000, 1 << 24), fields=rng.choice([1, 3, 4, 5, 8, 8, 12]),
                    p=round(math.exp(rng.uniform(math.log(0.0005), math.log(0.6))), 5))
    if kind == "tick":
        return dict(kind=kind, n=_log(rng, 1000, 1 << 23), fields=rng.choice([2, 4, 5, 8, 11]),
                    p=round(rng.uniform(0.005, 0.3), 4), mask=rng.random() < 0.4)
    if kind == "sort":
        return dict(kind=kind, n=_log(rng, 2000, 6_000_000), fields=rng.choice([1, 4, 5, 8]),
                    bits=rng.randint(6, 31), signed=rng.random() < 0.3, live=round(rng.uniform(0.1, 1.0), 3))
    if kind == "resolve":
        return dict(kind=kind, claims=_log(rng, 2000, 1 << 23), resources=_log(rng, 100, 1 << 20),
                    zipf=rng.choice([0.0, 0.8, 1.1, 1.3]))
    if kind == "match":
        cap = _log(rng, 60, 2048)
        return dict(kind=kind, books=_log(rng, 200, min(65536, (1 << 25) // cap)), cap=cap,
                    fill=round(rng.uniform(0.1, 0.9), 3), spread=rng.choice([5, 10, 40, 100]))
    if kind == "market":
        return dict(kind=kind, books=_log(rng, 10, 2000), cap=rng.randint(100, 1024), fill=round(rng.uniform(0, 0.4), 3),
                    traders=rng.randint(2, 20), steps=rng.randint(10, 100))
    if kind == "batch":
        lo = rng.randint(16, 64)
        return dict(kind=kind, models=_log(rng, 40, 2000), side_lo=lo, side_hi=rng.randint(lo + 16, 256),
                    steps=rng.randint(3, 30), warm=rng.randint(0, 60), extent=rng.random() < 0.5)
    return dict(kind=kind, rows=_log(rng, 2048, 32768), rows_per_step=rng.choice([256, 512, 1000, 1024]),
                hidden=rng.choice([64, 128, 128]), layers=rng.choice([2, 3, 3]))


# ---- what a program has in hand before the call


class _Device:
    """A slab's own device array, for torch.as_tensor (no copy); the tensor keeps it, and it keeps the slab."""

    def __init__(self, slab, address, shape):
        self.slab = slab
        self.__cuda_array_interface__ = dict(shape=shape, typestr="<i4", data=(address, False), version=2)


def _slab_views(s):
    """The slab's own arrays (live flags; fields, agent-major) as tensors."""
    import ctypes as C
    a, f, stride = C.c_void_p(), C.c_void_p(), C.c_int32()
    abm.call("abm_slab_arrays", s.h, C.byref(a), C.byref(f), C.byref(stride))
    return (torch.as_tensor(_Device(s, a.value, (s.capacity,)), device="cuda"),
            torch.as_tensor(_Device(s, f.value, (s.capacity, stride.value)), device="cuda")[:, :s.F])


def _ints(g, lo, hi, *shape):
    return torch.randint(lo, hi, shape, generator=g, device="cuda", dtype=torch.int64).to(torch.int32)


def _threshold(p):
    return int(p * 4294967296)


def _batch_models(case, seed):
    tab = workloads.sample_models(case["models"], seed % (1 << 31), case["side_lo"], case["side_hi"])
    caps = workloads.fixed_caps(tab["side"])
    return [dict(side=int(tab["side"][i]), seed=seed, model=i, params=tab["params"][i], cap=caps[i], n0=tab["n0"][i])
            for i in range(case["models"])]


def _books(case, g):
    n, cap, spread = case["books"], case["cap"], case.get("spread", 10)
    side = _ints(g, 0, 2, n, cap)
    price = torch.where(side == 0, 98 + (spread - 10), 102 + (spread - 10)) + _ints(g, -spread, spread + 1, n, cap)
    return dict(active=(torch.rand((n, cap), generator=g, device="cuda") < case["fill"]).to(torch.int32), side=side,
                price=price.to(torch.int32).clamp_(min=1), qty=_ints(g, 1, 101, n, cap),
                time=torch.argsort(torch.rand((n, cap), generator=g, device="cuda"), dim=1).to(torch.int32))


def _capacity_inputs(case, seed):
    """Features (on the scale of the library's), targets (log peak counts) and initial weights, float32 on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(seed)

    def uniform(lo, hi, *shape):
        return torch.rand(shape, generator=g, device="cuda") * (hi - lo) + lo
    n, h = case["rows"], case["hidden"]
    logs = uniform(2.8, 5.6, n, 1)
    x = torch.cat([logs, 2 * logs + uniform(-2.3, 0.7, n, 2), uniform(0.75, 1.25, n, 8), uniform(0.4, 1.0, n, 1)], 1)
    y = 2 * logs + uniform(-2.0, 1.0, n, 2)
    dims = [capacity.N_IN] + [h] * case["layers"] + [capacity.N_OUT]
    w = []
    for a, b in zip(dims[:-1], dims[1:]):
        w += [uniform(-1, 1, a * b) * math.sqrt(6.0 / a), torch.zeros(b, device="cuda")]
    return x.contiguous(), y.contiguous(), dims, torch.cat(w)


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    kind = case["kind"]
    st = dict(case=case, kind=kind, step=0)
    if kind == "world":
        w = engine.World(case["side"], seed, 0, workloads.predation_params(), (case["cap_sheep"], case["cap_wolves"]),
                         (case["sheep"], case["wolves"]), variant=case["variant"])
        if case["warm"]:
            w.step(case["warm"])
        st.update(world=w, stats=w.new_stats(case["steps"]))
        if case["resume"]:
            st["image"] = torch.zeros(w.image_bytes(), dtype=torch.uint8).pin_memory()
            w.save_into(st["image"])
            st["saved"] = torch.zeros(w.image_capacity(), dtype=torch.uint8).pin_memory()
        else:
            st["agents"] = [_slab_views(w.slab(s)) for s in range(2)]
    elif kind == "selective":
        n, F = case["n"], case["fields"]
        k = int(round(case["p"] * n))
        s = engine.Slab(n, F, seed=seed, init=abm.INIT_HALF_LIVE)
        st.update(slab=s, T=_threshold(case["p"]), records=_ints(g, -(1 << 31), 1 << 31, k, F),
                  deltas=_ints(g, -1000, 1000, k, F))
        for _ in range(8):  # the call's own steady state: free slots fill up over the first calls
            s.selective_update(st["step"], st["T"], st["records"], st["deltas"])
            st["step"] += 1
        st["views"] = _slab_views(s)
    elif kind == "tick":
        n, F = case["n"], case["fields"]
        k = max(1, int(case["p"] * n))
        s = engine.Slab(n, F, seed=seed, init=abm.INIT_HALF_LIVE)
        for f in range(F):
            s.write(f, _ints(g, 0, 1000, n))
        st.update(slab=s, k=k, newborn=_ints(g, 0, 1000, k, F), change=_ints(g, -9, 10, k, F),
                  mask=_ints(g, 0, 2, k) if case["mask"] else None, who=torch.full((n,), -1, dtype=torch.int32, device="cuda"),
                  slots=torch.full((2, k), -1, dtype=torch.int32, device="cuda"),
                  counts=torch.zeros(4, dtype=torch.int32, device="cuda"), views=_slab_views(s))
    elif kind == "sort":
        n = case["n"]
        s = engine.Slab(n, case["fields"], seed=seed, init=abm.INIT_HALF_LIVE)
        lo = -(1 << (case["bits"] - 1)) if case["signed"] else 0
        st.update(slab=s, keys=_ints(g, lo, lo + (1 << case["bits"]), n),
                  live=(torch.rand(n, generator=g, device="cuda") < case["live"]).to(torch.int32))
    elif kind == "resolve":
        M, R = case["claims"], case["resources"]
        cdf = torch.cumsum(torch.arange(1, R + 1, dtype=torch.float64, device="cuda") ** -case["zipf"], 0)
        u = torch.rand(M, generator=g, device="cuda", dtype=torch.float64) * cdf[-1]
        st.update(resolver=engine.Resolver(R), res=torch.searchsorted(cdf, u).clamp_(max=R - 1).to(torch.int32),
                  prio=_ints(g, -(1 << 31), 1 << 31, M), won=torch.zeros(M, dtype=torch.uint8, device="cuda"))
    elif kind == "match":
        books = engine.OrderBooks(_books(case, g))
        st.update(books=books, opening={f: books.t[f].clone() for f in ("active", "qty")})
    elif kind == "market":
        n, K, S = case["books"], case["traders"], case["steps"]
        books = engine.OrderBooks(_books(case, g))
        side = _ints(g, 0, 2, S, n, K)
        price = torch.where(side == 0, 98, 102) + _ints(g, -10, 11, S, n, K)
        time = (torch.arange(S * K, device="cuda").reshape(S, 1, K) + (1 << 20)).expand(S, n, K)
        orders = torch.stack([side, price.to(torch.int32), _ints(g, 1, 101, S, n, K), time.to(torch.int32)], 3).contiguous()
        ks = _ints(g, 0, K + 1, S, n)
        opening = {f: t.clone() for f, t in books.t.items()}
        volume = torch.zeros((S, n), dtype=torch.int64, device="cuda")
        price, added = (torch.zeros((S, n), dtype=torch.int32, device="cuda") for _ in range(2))

        def session():
            for f, t in books.t.items():
                t.copy_(opening[f])
            for i in range(S):
                books.add(orders[i], ks[i], out=added[i])
                books.match(out_volume=volume[i], out_price=price[i])
        session()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            session()
        st.update(graph=graph, keep=(orders, ks, opening), out=[books.t[f] for f in books.FIELDS] + [volume, price, added])
    elif kind == "batch":
        b = engine.Batch(_batch_models(case, seed))
        cells = case["side_hi"] ** 2  # room for the first model's state, whatever its side
        st.update(batch=b, sweep=abm.SWEEP_EXTENT if case["extent"] else abm.SWEEP_CAPACITY,
                  agents=torch.zeros((2, len(engine.AGENT_FIELDS), 4 * cells), dtype=torch.int32, device="cuda"),
                  grass=torch.zeros(cells, dtype=torch.int32, device="cuda"))
        if case["warm"]:
            b.run(case["warm"], sweep=abm.SWEEP_EXTENT)
    else:
        x, y, _, w = _capacity_inputs(case, seed)
        m = capacity.CapacityModel(workloads.predation_params(), hidden=case["hidden"], layers=case["layers"],
                                   seed=seed % 1000)
        m.set_params(w)
        st.update(model=m, x=x, y=y)
    return st


# ---- one pass


def run(st):
    case, kind = st["case"], st["kind"]
    if kind == "world":
        w = st["world"]
        if case["resume"]:
            w.load_from(st["image"])
            w.step(case["steps"], stats=st["stats"])
            w.save_into(st["saved"])
            return [st["stats"], st["saved"]]
        w.step(case["steps"], stats=st["stats"])
        return [st["stats"], w.grass("wait")] + [t for views in st["agents"] for t in views]
    if kind == "selective":
        counts = st["slab"].selective_update(st["step"], st["T"], st["records"], st["deltas"])
        st["step"] += 1
        return [counts, *st["views"]]
    if kind == "tick":
        s, F, k, T = st["slab"], case["fields"], st["k"], _threshold(case["p"])
        stream, ptr, ref, n = abm.stream_handle(), abm.ptr, abm.C.byref, st["counts"]
        st["step"] += 1
        hungry = abm.pred(abm.PRED_FIELD, field=0, cmp=abm.CMP_LT, value=100)
        moved = abm.pred(abm.PRED_BERNOULLI, threshold=T, step=st["step"], purpose=abm.P_MOVE)
        dying = abm.pred(abm.PRED_BERNOULLI, threshold=T, step=st["step"], purpose=abm.P_REPRO)
        abm.call("abm_select", s.h, ref(hungry), ptr(st["who"]), ptr(n[0:]), stream)
        abm.call("abm_update_distinct", s.h, ref(moved), ptr(st["change"]), ptr(st["mask"]), k, abm.OP_ADD,
                 ptr(st["slots"][0]), ptr(n[1:]), stream)
        abm.call("abm_remove", s.h, ref(dying), ptr(n[2:]), stream)
        abm.call("abm_add", s.h, ptr(st["newborn"]), k, F - 1, ptr(st["slots"][1]), ptr(n[3:]), stream)
        return [n, st["who"], st["slots"], *st["views"]]
    if kind == "sort":
        s = st["slab"]
        s.write(0, st["keys"])
        s.write(-1, st["live"])
        order = s.sort(0)
        return [order, *_slab_views(s)]
    if kind == "resolve":
        return [st["resolver"](st["res"], st["prio"], is_winner=st["won"]), st["won"]]
    if kind == "match":
        books = st["books"]
        for f, t in st["opening"].items():
            books.t[f].copy_(t)
        volume, price = books.match()
        return [volume, price, books.t["active"], books.t["qty"]]
    if kind == "market":
        st["graph"].replay()
        return st["out"]
    if kind == "batch":
        b = st["batch"]
        b.run(case["steps"], sweep=st["sweep"])
        for s in range(2):
            for f in range(len(engine.AGENT_FIELDS)):
                abm.call("abm_batch_read_agents", b.h, 0, s, f, abm.ptr(st["agents"][s][f]), abm.stream_handle())
        abm.call("abm_batch_read_grass", b.h, 0, 1, abm.ptr(st["grass"]), abm.stream_handle())
        return [b.digest(), st["agents"], st["grass"]]  # every model's state digest, the first model's whole state
    m = st["model"]
    m.fit(st["x"], st["y"], epochs=1, batch=case["rows_per_step"])
    return [m.params(), m.grads(), m.predict(st["x"])]


# ---- what a pass cannot do without


def work(case):
    kind = case["kind"]
    if kind == "world":  # records of live agents in and out, their flags, a grass word per sheep, stats
        a = case["sheep"] + case["wolves"]
        b = case["steps"] * (a * 36 + case["sheep"] * 4 + abm.STATS_BYTES)
        if case["resume"]:
            b += 2 * (a * 20 + case["side"] ** 2 * 4)
        return dict(bytes=b, flops=0)
    if kind == "selective":  # flags in; per removed / added / updated agent its flag, record and row
        n, row = case["n"], 4 * case["fields"]
        k = int(round(case["p"] * n))
        return dict(bytes=4 * n + k * (4 + 4 + 2 * row + (1 - case["p"]) * 3 * row), flops=0)
    if kind == "tick":
        n, row, k = case["n"], 4 * case["fields"], int(case["p"] * case["n"])
        return dict(bytes=4 * n * 2 + 0.1 * n * 4 + k * (5 * row + 16), flops=0)
    if kind == "sort":  # new keys and flags in; rows, flags and the permutation
        return dict(bytes=case["n"] * (8 + 2 * (4 * case["fields"] + 4) + 4), flops=0)
    if kind == "resolve":
        return dict(bytes=case["claims"] * 9 + case["resources"] * 4, flops=0)
    if kind == "match":  # flags in, the live orders' words, changed flags and quantities; the opening's two arrays
        n = case["books"] * case["cap"]
        return dict(bytes=n * (16 + 4 + 12 * case["fill"] + 8 * case["fill"]) + 12 * case["books"], flops=0)
    if kind == "market":
        n = case["books"] * case["cap"]
        return dict(bytes=n * 40 + case["steps"] * (n * (4 + 12 * case["fill"]) + case["books"] * (16 * case["traders"] + 20)), flops=0)
    if kind == "batch":  # per step: flags of every slot (static shapes) or of the live ones, live records in and out
        cells = case["models"] * (case["side_lo"] ** 2 + case["side_lo"] * case["side_hi"] + case["side_hi"] ** 2) / 3
        slots = cells * (1.0 if case["extent"] else 8.0)
        return dict(bytes=case["steps"] * (slots * 4 + cells * 0.35 * 36), flops=0)
    n, h = case["rows"], case["hidden"]
    params = 12 * h + h * h * (case["layers"] - 1) + 2 * h
    steps = n // case["rows_per_step"]
    return dict(bytes=n * 2 * 56 + steps * params * 28, flops=n * params * 8)


# ---- the same in 64 bits


def exact(case, seed):
    """The predictor's epoch in float64 (everything else is whole numbers and bytes)."""
    if case["kind"] != "capacity":
        return None
    x, y, dims, w = _capacity_inputs(case, seed)
    x, y, w = x.double(), y.double(), w.double()
    n, B, tau, lr = case["rows"], case["rows_per_step"], 0.99, 1e-3
    rng = np.random.default_rng(seed % 1000)  # the epoch's order: row = (a * i + c) mod n
    while True:
        a = int(rng.integers(1, n)) | 1
        if np.gcd(a, n) == 1:
            break
    c = int(rng.integers(0, n))

    def layers(flat):
        at = 0
        for p, q in zip(dims[:-1], dims[1:]):
            yield flat[at:at + p * q].view(p, q), flat[at + p * q:at + p * q + q]
            at += p * q + q

    def forward(x, flat):
        for i, (W, b) in enumerate(layers(flat)):
            x = x @ W + b
            x = torch.relu(x) if i < len(dims) - 2 else x
        return x
    m, v, grad = torch.zeros_like(w), torch.zeros_like(w), torch.zeros_like(w)
    for t, i0 in enumerate(range(0, n - B + 1, B), 1):
        rows = (a * torch.arange(i0, i0 + B, device="cuda") + c) % n
        w = w.detach().requires_grad_()
        e = y[rows] - forward(x[rows], w)
        torch.where(e > 0, tau * e, (tau - 1) * e).mean().backward()
        grad = w.grad
        m, v = 0.9 * m + 0.1 * grad, 0.999 * v + 0.001 * grad * grad
        w = w.detach() - lr * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)
    w = w.detach()
    return [w, grad, forward(x, w)]
