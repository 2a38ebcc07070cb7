"""GPU parity: generic slab primitives and conflict resolution vs the oracle.

Every comparison is element by element and bit-exact (all arithmetic is
integer). Sizes span several 2048-slot tiles plus ragged tails, and the
selective-update microbenchmark is also checked at its full size (2^24 slots
x 8 fields) against the oracle on the same seeded inputs.
"""
import numpy as np
import pytest

import oracle
import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eng():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2508_16508_gb300 import abm, engine
    abm.lib()
    return engine


def np_of(t):
    return t.cpu().numpy()


def slab_state(s):
    torch.cuda.synchronize()
    return np_of(s.read(-1)), np.stack([np_of(s.read(f)) for f in range(s.F)])


SIZES = [1, 3, 33, 2047, 2048, 2049, 4096 * 3 + 17, 100_003]


@pytest.mark.parametrize("n", SIZES)
def test_half_live_init(eng, n):
    s = eng.Slab(n, 8, seed=2, init=1)
    o = oracle.Slab(n, 8)
    o.c1_init(seed=2)
    act, fld = slab_state(s)
    np.testing.assert_array_equal(act, o.active)
    np.testing.assert_array_equal(fld, o.fields)
    assert s.counters()["n_active"] == int(o.active.sum())


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("p", [0.001, 0.05, 0.5])
def test_selective_update_parity(eng, n, p):
    from paper_2508_16508_gb300 import abm
    F = 8
    T, k = workloads.threshold(p), max(workloads.k_for(p, n), 1)
    s = eng.Slab(n, F, seed=2, init=1)
    o = oracle.Slab(n, F)
    o.c1_init(seed=2)
    for step in range(4):
        rec = s.philox_records(step, abm.P_NEWREC0, abm.P_NEWREC1, k)
        dl = s.philox_records(step, abm.P_DELTA0, abm.P_DELTA1, k)
        np.testing.assert_array_equal(np_of(rec), oracle.c1_records(2, 0, step, oracle.P_NEWREC0,
                                                                    oracle.P_NEWREC1, k, F))
        cnt = np_of(s.selective_update(step, T, rec, dl))
        want = o.c1_call(step, T, k, seed=2)
        act, fld = slab_state(s)
        s.check()
        assert cnt.tolist() == [want["removed"], want["added"], want["updated"]]
        np.testing.assert_array_equal(act, o.active)
        np.testing.assert_array_equal(fld, o.fields)
        assert s.counters()["n_active"] == int(o.active.sum())


@pytest.mark.parametrize("offset", [0, 4, 1])
@pytest.mark.parametrize("p", [0.05, 0.5])
def test_selective_update_record_alignment(eng, offset, p):
    """Records and deltas starting 0, 16 or 4 bytes past a 32-byte boundary
    (the three ways the apply pass moves 8-field rows) give the same slab."""
    from paper_2508_16508_gb300 import abm
    n, F = 20_011, 8
    T, k = workloads.threshold(p), workloads.k_for(p, n)
    s = eng.Slab(n, F, seed=4, init=1)
    o = oracle.Slab(n, F)
    o.c1_init(seed=4)
    rb = torch.empty(k * F + 8, dtype=torch.int32, device="cuda")
    db = torch.empty(k * F + 8, dtype=torch.int32, device="cuda")
    rec, dl = rb[offset:offset + k * F].view(k, F), db[offset:offset + k * F].view(k, F)
    for step in range(3):
        s.philox_records(step, abm.P_NEWREC0, abm.P_NEWREC1, k, out=rec)
        s.philox_records(step, abm.P_DELTA0, abm.P_DELTA1, k, out=dl)
        cnt = np_of(s.selective_update(step, T, rec, dl))
        want = o.c1_call(step, T, k, seed=4)
        assert cnt.tolist() == [want["removed"], want["added"], want["updated"]]
        act, fld = slab_state(s)
        np.testing.assert_array_equal(act, o.active)
        np.testing.assert_array_equal(fld, o.fields)
    s.check()


def test_live_flag_values(eng):
    """Nonzero flags other than 1 count as live everywhere; a call that fills a
    16-slot group (add) or empties an 8-slot group (the fused call) writes that
    group's flags as 0/1, and every other flag keeps its value."""
    from paper_2508_16508_gb300 import abm
    n, F = 4000, 3
    rng = np.random.default_rng(8)
    flags = np.where(rng.random(n) < 0.7, rng.choice([1, 7, -2], size=n), 0).astype(np.int32)
    s = eng.Slab(n, F)
    s.write(-1, torch.from_numpy(flags).cuda())
    o = oracle.Slab(n, F)
    o.active[:] = flags != 0
    k = 40
    rec = rng.integers(-9, 9, size=(k, F)).astype(np.int32)
    slots, cnt = s.add(torch.from_numpy(rec).cuda())
    r, want_slots = o.add(rec)
    assert int(cnt.item()) == r == k
    np.testing.assert_array_equal(np_of(slots[:r]), want_slots)
    got = np_of(s.read(-1))
    np.testing.assert_array_equal(got != 0, o.active != 0)
    filled = np.zeros(n, bool)
    for g in np.unique(want_slots // 16):
        filled[16 * g:16 * g + 16] = True
    assert set(np.unique(got[filled]).tolist()) <= {0, 1}
    np.testing.assert_array_equal(got[~filled], flags[~filled])
    # a mask array that starts 4 bytes past an aligned address (scalar loads)
    buf = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
    tm = (rng.random(n) < 0.5).astype(np.int32)
    buf[1:] = torch.from_numpy(tm).cuda()
    d = rng.integers(-5, 5, size=(300, F)).astype(np.int32)
    rmask = torch.zeros(301, dtype=torch.int32, device="cuda")
    rm = (rng.random(300) < 0.5).astype(np.int32)
    rmask[1:] = torch.from_numpy(rm).cuda()
    _, ucnt = s.update_distinct(abm.pred(abm.PRED_MASK, mask=buf[1:]), torch.from_numpy(d).cuda(),
                                rmask[1:], op=abm.OP_ADD)
    ru, _ = o.update_distinct(tm.astype(bool) & (o.active != 0), d, rec_mask=rm, op=0)
    assert int(ucnt.item()) == ru
    _, fld = slab_state(s)
    np.testing.assert_array_equal(fld, o.fields)
    s.check()


def test_selective_update_equals_separate_calls(eng):
    from paper_2508_16508_gb300 import abm
    n, F, p = 50_000, 8, 0.05
    T, k = workloads.threshold(p), workloads.k_for(p, n)
    a = eng.Slab(n, F, seed=5, init=1)
    b = eng.Slab(n, F, seed=5, init=1)
    for step in range(3):
        rec = a.philox_records(step, abm.P_NEWREC0, abm.P_NEWREC1, k)
        dl = a.philox_records(step, abm.P_DELTA0, abm.P_DELTA1, k)
        a.selective_update(step, T, rec, dl)
        # the same call as remove -> distinct update -> add through the generic API,
        # with the two draws made into explicit masks
        # slots 2j and 2j+1 share draw j: words (0, 1) and (2, 3) = (remove, choose)
        w = np.stack([oracle.philox_words(5, 0, step, oracle.P_MASK, 0, 0, (n + 1) // 2, q)
                      for q in range(4)]).astype(np.int64)
        slot = np.arange(n)
        rm = torch.from_numpy((w[2 * (slot & 1), slot >> 1] < T).astype(np.int32)).cuda()
        ch = torch.from_numpy((w[2 * (slot & 1) + 1, slot >> 1] < T).astype(np.int32)).cuda()
        b.remove(abm.pred(abm.PRED_MASK, mask=rm))
        b.update_distinct(abm.pred(abm.PRED_MASK, mask=ch), dl, op=abm.OP_ADD)
        b.add(rec)
        for f in range(-1, F):
            assert torch.equal(a.read(f), b.read(f))


def test_selective_update_full_size(eng):
    """2^24 slots x 8 fields, all three p, three calls each: full-state parity."""
    from paper_2508_16508_gb300 import abm
    c = workloads.SELECTIVE
    n, F = c["n"], c["F"]
    for p in c["p"]:
        T, k = workloads.threshold(p), workloads.k_for(p, n)
        s = eng.Slab(n, F, seed=c["seed"], init=1)
        o = oracle.Slab(n, F)
        o.c1_init(seed=c["seed"])
        for step in range(3):
            rec = s.philox_records(step, abm.P_NEWREC0, abm.P_NEWREC1, k)
            dl = s.philox_records(step, abm.P_DELTA0, abm.P_DELTA1, k)
            cnt = np_of(s.selective_update(step, T, rec, dl))
            want = o.c1_call(step, T, k, seed=c["seed"])
            assert cnt.tolist() == [want["removed"], want["added"], want["updated"]]
        act, fld = slab_state(s)
        s.check()
        np.testing.assert_array_equal(act, o.active)
        np.testing.assert_array_equal(fld, o.fields)
        del s


@pytest.mark.parametrize("n", [1, 31, 2048, 2049, 9000])
def test_select_predicates(eng, n):
    from paper_2508_16508_gb300 import abm
    s = eng.Slab(n, 3, seed=9, init=1)
    act, fld = slab_state(s)
    rng = np.random.default_rng(n)
    mask = (rng.random(n) < 0.3).astype(np.int32)
    cases = [
        (abm.pred(abm.PRED_LIVE), act != 0),
        (abm.pred(abm.PRED_FREE), act == 0),
        (abm.pred(abm.PRED_BERNOULLI, threshold=workloads.threshold(0.25), step=4, purpose=abm.P_REPRO),
         (act != 0) & (oracle.philox_words(9, 0, 4, oracle.P_REPRO, 0, 0, n) < workloads.threshold(0.25))),
        (abm.pred(abm.PRED_MASK, mask=torch.from_numpy(mask).cuda()), (act != 0) & (mask != 0)),
        (abm.pred(abm.PRED_FIELD, field=1, cmp=abm.CMP_EQ, and_mask=1, value=0),
         (act != 0) & ((fld[1] & 1) == 0)),
        (abm.pred(abm.PRED_FIELD, field=2, cmp=abm.CMP_LT, value=0), (act != 0) & (fld[2] < 0)),
        (abm.pred(abm.PRED_FIELD, field=0, cmp=abm.CMP_GE, value=12345), (act != 0) & (fld[0] >= 12345)),
        (abm.pred(abm.PRED_FIELD, field=0, cmp=abm.CMP_NE, and_mask=3, value=2),
         (act != 0) & ((fld[0] & 3) != 2)),
    ]
    for p, want_mask in cases:
        idx, cnt = s.select(p)
        c = int(cnt.item())
        want = oracle.flatnonzero(want_mask.astype(np.int32))
        assert c == want.size
        np.testing.assert_array_equal(np_of(idx[:c]), want)


@pytest.mark.parametrize("n", [1, 33, 2049, 4096 * 3 + 17])
def test_select_permutation(eng, n):
    """SCI's index exposure (Algorithm 2): the selected slots ascending, then
    the rest ascending -- the stable argsort of the mask with true first."""
    from paper_2508_16508_gb300 import abm
    s = eng.Slab(n, 3, seed=6, init=1)
    act, fld = slab_state(s)
    T = workloads.threshold(0.5)
    cases = [(abm.pred(abm.PRED_LIVE), act != 0),
             (abm.pred(abm.PRED_FREE), act == 0),
             (abm.pred(abm.PRED_BERNOULLI, threshold=T, step=3, purpose=abm.P_REPRO, species=1),
              (act != 0) & (oracle.philox_words(6, 0, 3, oracle.P_REPRO, 1, 0, n) < T)),
             (abm.pred(abm.PRED_FIELD, field=2, cmp=abm.CMP_LT, and_mask=0xFF, value=100),
              (act != 0) & ((fld[2] & 0xFF) < 100))]
    for p, m in cases:
        perm, cnt = s.select_permutation(p)
        sel = oracle.flatnonzero(m.astype(np.int32))
        rest = oracle.flatnonzero((~m).astype(np.int32))
        assert int(cnt.item()) == sel.size
        np.testing.assert_array_equal(np_of(perm), np.concatenate([sel, rest]))
        np.testing.assert_array_equal(np_of(perm), np.argsort(~m, kind="stable"))
    s.check()


@pytest.mark.parametrize("n", [1, 33, 2049, 4096 * 3 + 17, 100_003])
def test_sort_agents(eng, n):
    """sort_agents vs the oracle: whole state and permutation, keys with many
    ties (stability) and full-range keys, twice in a row (the second call
    sorts by another field and reuses the buffers)."""
    F = 5
    rng = np.random.default_rng(n)
    s = eng.Slab(n, F, seed=4, init=1)
    o = oracle.Slab(n, F)
    o.c1_init(seed=4)
    ties = rng.integers(-3, 4, size=n).astype(np.int32)
    s.write(1, torch.from_numpy(ties).cuda())
    o.fields[1] = ties
    for field in (1, 3, 0):
        perm = np_of(s.sort(field))
        want = o.sort(field)
        np.testing.assert_array_equal(perm, want)
        act, fld = slab_state(s)
        np.testing.assert_array_equal(act, o.active)
        np.testing.assert_array_equal(fld, o.fields)
    assert s.counters()["n_active"] == int(o.active.sum())
    # live flags other than 0 / 1 (written by the caller) move unchanged
    odd = np.where(o.active != 0, 7, 0).astype(np.int32)
    s.write(-1, torch.from_numpy(odd).cuda())
    o.active[:] = odd
    np.testing.assert_array_equal(np_of(s.sort(2)), o.sort(2))
    act, fld = slab_state(s)
    np.testing.assert_array_equal(act, o.active)
    np.testing.assert_array_equal(fld, o.fields)
    s.check()


def test_maximum_capacity(eng):
    """The largest slab abm_slab_create accepts (2^28 - 1 slots, one field):
    half-live init, one selective-update call and a select, against the
    oracle; then a sort by the field."""
    from paper_2508_16508_gb300 import abm
    n, F, p = (1 << 28) - 1, 1, 0.001
    T, k = workloads.threshold(p), workloads.k_for(p, n)
    s = eng.Slab(n, F, seed=8, init=1)
    o = oracle.Slab(n, F)
    o.c1_init(seed=8)
    rec = s.philox_records(0, abm.P_NEWREC0, abm.P_NEWREC1, k)
    dl = s.philox_records(0, abm.P_DELTA0, abm.P_DELTA1, k)
    cnt = np_of(s.selective_update(0, T, rec, dl))
    want = o.c1_call(0, T, k, seed=8)
    assert cnt.tolist() == [want["removed"], want["added"], want["updated"]]
    act, fld = slab_state(s)
    np.testing.assert_array_equal(act, o.active)
    np.testing.assert_array_equal(fld, o.fields)
    del act, fld
    idx, c = s.select(abm.pred(abm.PRED_LIVE))
    live = int(c.item())
    assert live == int(o.active.sum()) == s.counters()["n_active"]
    assert bool((idx[1:live] > idx[:live - 1]).all())
    del idx
    # the sort, by the properties that define it (the oracle's sort is O(n log n)
    # on one core; the small and 2^24 cases compare with it directly)
    act0, key0 = o.active, o.fields[0]
    perm = np_of(s.sort(0)).astype(np.int64)
    assert (np.bincount(perm, minlength=n) == 1).all()  # a permutation
    act, fld = slab_state(s)
    np.testing.assert_array_equal(act, act0[perm])
    np.testing.assert_array_equal(fld[0], key0[perm])
    assert (act[:live] != 0).all() and (act[live:] == 0).all()
    k = fld[0][:live].astype(np.int64)
    pl = perm[:live]
    assert ((k[1:] > k[:-1]) | ((k[1:] == k[:-1]) & (pl[1:] > pl[:-1]))).all()  # ascending, stable
    assert (np.diff(perm[live:]) > 0).all()  # placeholders in slot order
    s.check()


def test_sort_agents_full_size(eng):
    """2^24 slots x 8 fields (the selective-update slab), after three
    selective-update calls; sorted by two fields."""
    from paper_2508_16508_gb300 import abm
    c = workloads.SELECTIVE
    n, F, p = c["n"], c["F"], 0.05
    T, k = workloads.threshold(p), workloads.k_for(p, n)
    s = eng.Slab(n, F, seed=c["seed"], init=1)
    o = oracle.Slab(n, F)
    o.c1_init(seed=c["seed"])
    for step in range(3):
        rec = s.philox_records(step, abm.P_NEWREC0, abm.P_NEWREC1, k)
        dl = s.philox_records(step, abm.P_DELTA0, abm.P_DELTA1, k)
        s.selective_update(step, T, rec, dl)
        o.c1_call(step, T, k, seed=c["seed"])
    for field in (2, 7):
        np.testing.assert_array_equal(np_of(s.sort(field)), o.sort(field))
    act, fld = slab_state(s)
    np.testing.assert_array_equal(act, o.active)
    np.testing.assert_array_equal(fld, o.fields)
    s.check()


@pytest.mark.parametrize("n", [5, 2049, 7000])
def test_add_remove_update_vs_oracle(eng, n):
    from paper_2508_16508_gb300 import abm
    F = 5
    rng = np.random.default_rng(n)
    s = eng.Slab(n, F)
    o = oracle.Slab(n, F)
    next_id = 0
    for it in range(6):
        k = int(rng.integers(0, n // 2 + 2))
        rec = rng.integers(-2**31, 2**31, size=(k, F), dtype=np.int64).astype(np.int32)
        slots, cnt = s.add(torch.from_numpy(rec).cuda(), id_field=4)
        r, want_slots = o.add(rec, id_field=4, id_base=next_id)
        next_id += r
        assert int(cnt.item()) == r
        np.testing.assert_array_equal(np_of(slots[:r]), want_slots)
        m = (rng.random(n) < 0.2).astype(np.int32)
        rem = s.remove(abm.pred(abm.PRED_MASK, mask=torch.from_numpy(m).cuda()))
        assert int(rem.item()) == o.remove(m)
        tm = (rng.random(n) < 0.4).astype(np.int32)
        kd = int(rng.integers(0, n // 3 + 2))
        d = rng.integers(-2**31, 2**31, size=(kd, F), dtype=np.int64).astype(np.int32)
        rm = (rng.random(kd) < 0.6).astype(np.int32) if it % 2 else None
        op = abm.OP_ADD if it % 3 else abm.OP_SET
        us, ucnt = s.update_distinct(abm.pred(abm.PRED_MASK, mask=torch.from_numpy(tm).cuda()),
                                     torch.from_numpy(d).cuda(),
                                     None if rm is None else torch.from_numpy(rm).cuda(), op=op)
        ru, want_us = o.update_distinct(tm.astype(bool) & o.active.astype(bool), d, rec_mask=rm, op=op)
        assert int(ucnt.item()) == ru
        np.testing.assert_array_equal(np_of(us[:ru]), want_us)
        act, fld = slab_state(s)
        np.testing.assert_array_equal(act, o.active)
        np.testing.assert_array_equal(fld, o.fields)
        assert s.counters()["n_active"] == int(o.active.sum())
        assert s.counters()["next_id"] == next_id
    s.check()


def test_add_overflow_flag(eng):
    s = eng.Slab(10, 2)
    slots, cnt = s.add(torch.arange(24, dtype=torch.int32, device="cuda").reshape(12, 2))
    assert int(cnt.item()) == 10
    c = s.counters()
    assert c["overflow"] == 1 and c["n_active"] == 10


def test_toy_task_on_gpu(eng):
    """Section 4's toy task through update_distinct (SET) with both masks."""
    from paper_2508_16508_gb300 import abm
    import os
    d = {}
    with open(os.path.join(os.path.dirname(__file__), "golden", "toy_task.txt")) as f:
        for line in f:
            if line.strip() and not line.startswith("#"):
                k, v = line.split(":")
                d[k.strip()] = [int(x) for x in v.split()]
    a, b = d["a"], d["b"]
    s = eng.Slab(len(a), 1)
    s.add(torch.tensor(a, dtype=torch.int32, device="cuda").reshape(-1, 1))
    bt = torch.tensor(b, dtype=torch.int32, device="cuda").reshape(-1, 1)
    _, cnt = s.update_distinct(abm.pred(abm.PRED_FIELD, field=0, cmp=abm.CMP_EQ, and_mask=1, value=0),
                               bt, record_mask=(bt[:, 0] & 1), op=abm.OP_SET)
    assert int(cnt.item()) == d["r"][0]
    assert np_of(s.read(0)).tolist() == d["expected"]


@pytest.mark.parametrize("M,R", [(0, 5), (1, 1), (1000, 7), (4097, 300), (100_000, 65_536), (300_001, 1024)])
def test_resolve_vs_oracle(eng, M, R):
    rng = np.random.default_rng(M + R)
    res = rng.integers(-2, R + 2, size=M).astype(np.int32)
    if M > 10:
        res[: M // 3] = workloads.zipf_claims(M // 3, R, seed=M)
    prio = rng.integers(0, 8, size=M).astype(np.uint32) * np.uint32(0x20000000)
    r = eng.Resolver(R)
    isw = torch.empty(max(M, 1), dtype=torch.uint8, device="cuda")
    dres = torch.from_numpy(res).cuda()
    dprio = torch.from_numpy(prio.view(np.int32)).cuda()
    for rep in range(2):  # the scratch table must come back clean
        w = r(dres, dprio, isw[:M] if M else None)
        ow, oisw = oracle.resolve(res, prio, R)
        np.testing.assert_array_equal(np_of(w), ow)
        if M:
            np.testing.assert_array_equal(np_of(isw[:M]), oisw)
    assert torch.all(r.table == -1)


def test_resolve_full_size(eng):
    c = workloads.SELECTIVE
    N = c["n"]
    M, R = N // 4, N // 64
    res = workloads.zipf_claims(M, R, s=c["zipf_s"], seed=c["zipf_seed"])
    prio = oracle.philox_words(c["seed"], 0, 0, oracle.P_RESOURCE, 0, 0, M)
    r = eng.Resolver(R)
    isw = torch.empty(M, dtype=torch.uint8, device="cuda")
    w = r(torch.from_numpy(res).cuda(), torch.from_numpy(prio.view(np.int32)).cuda(), isw)
    ow, oisw = oracle.resolve(res, prio, R)
    np.testing.assert_array_equal(np_of(w), ow)
    np.testing.assert_array_equal(np_of(isw), oisw)


def test_argument_errors(eng):
    from paper_2508_16508_gb300 import abm
    import ctypes as C
    h = C.c_void_p()
    L = abm.lib()
    assert L.abm_slab_create(0, 8, 0, 0, 0, None, C.byref(h)) == abm.ERR_ARG
    assert L.abm_slab_create(10, 17, 0, 0, 0, None, C.byref(h)) == abm.ERR_ARG
    assert L.abm_slab_create(1 << 28, 1, 0, 0, 0, None, C.byref(h)) == abm.ERR_ARG
    assert L.abm_resolve(None, None, 5, 3, None, None, None, None) == abm.ERR_ARG
    s = eng.Slab(10, 2)
    assert L.abm_select(s.h, None, None, None, None) == abm.ERR_ARG
    p = abm.pred(abm.PRED_FIELD, field=2)
    assert L.abm_select(s.h, C.byref(p), None, None, None) == abm.ERR_ARG


@pytest.mark.parametrize("n,F", [(1, 1), (33, 3), (4097, 16), (16_384, 4), (16_385, 9), (20_481, 5), (700_001, 2)])
@pytest.mark.parametrize("keys", ["equal", "byte2", "signed", "all_bits", "none_live", "all_live"])
def test_sort_agents_key_ranges(eng, n, F, keys):
    """Whole numbers, so exact: keys whose bytes are all alike (their passes are left out), in every position,
    negative keys, all bits, and no or only live agents, at the edges of the sort's tiles."""
    rng = np.random.default_rng(n + F)
    k = {"equal": np.full(n, -7), "byte2": rng.integers(0, 40, n) << 16, "signed": rng.integers(-300, 300, n),
         "all_bits": rng.integers(-2**31, 2**31, n)}.get(keys, rng.integers(0, 1000, n)).astype(np.int32)
    live = {"none_live": np.zeros(n), "all_live": np.ones(n)}.get(keys, rng.random(n) < 0.6).astype(np.int32)
    rest = rng.integers(-2**31, 2**31, (F, n)).astype(np.int32)
    field = F - 1
    rest[field] = k
    s = eng.Slab(n, F)
    for f in range(F):
        s.write(f, torch.from_numpy(rest[f]).cuda())
    s.write(-1, torch.from_numpy(live).cuda())
    assert s.counters()["n_active"] == int(live.sum())
    want = np.lexsort((np.arange(n), np.where(live, k, 0), live == 0))
    np.testing.assert_array_equal(np_of(s.sort(field)), want)
    np.testing.assert_array_equal(np_of(s.read(-1)), live[want])
    for f in range(F):
        np.testing.assert_array_equal(np_of(s.read(f)), rest[f][want])


@pytest.mark.parametrize("n", [1, 31, 4097, 65_536, 65_537, 131_072, 131_073, 200_001, 262_144, 262_145])
@pytest.mark.parametrize("F", [1, 3, 8, 12])
def test_one_launch_sizes(eng, n, F):
    """Whole numbers, so exact: every set operation at the sizes where the one-launch path changes its slots per lane
    and its cluster, and one slot past it, against the operations written out with numpy; flags other than 0 and 1."""
    from paper_2508_16508_gb300 import abm
    rng = np.random.default_rng(n * 16 + F)
    s = eng.Slab(n, F, seed=9)
    act = np.where(rng.random(n) < 0.5, rng.choice([1, 1, 1, 7], n), 0).astype(np.int32)
    fld = rng.integers(-50, 50, (F, n)).astype(np.int32)
    s.write(-1, torch.from_numpy(act).cuda())
    for f in range(F):
        s.write(f, torch.from_numpy(fld[f]).cuda())
    k = max(1, n // 7)
    rec = rng.integers(-2**31, 2**31, (k, F)).astype(np.int32)
    rmask = (rng.random(k) < 0.5).astype(np.int32)
    dev = torch.from_numpy(rec).cuda()

    def check(where):
        np.testing.assert_array_equal(np_of(s.read(-1)) != 0, act != 0, err_msg=where)
        for f in range(F):
            np.testing.assert_array_equal(np_of(s.read(f)), fld[f], err_msg=where)
        assert s.counters()["n_active"] == int((act != 0).sum()), where

    p = abm.pred(abm.PRED_FIELD, field=F - 1, cmp=abm.CMP_LT, value=0)
    idx, cnt = s.select(p)
    want = np.flatnonzero((act != 0) & (fld[F - 1] < 0))
    np.testing.assert_array_equal(np_of(idx)[:int(cnt)], want)
    perm, cnt = s.select_permutation(p)
    sel = (act != 0) & (fld[F - 1] < 0)
    np.testing.assert_array_equal(np_of(perm), np.argsort(~sel, kind="stable"))
    for masked, op in ((False, abm.OP_ADD), (True, abm.OP_SET)):
        p = abm.pred(abm.PRED_FIELD, field=0, cmp=abm.CMP_GE, value=-10)
        sel = np.flatnonzero((act != 0) & (fld[0] >= -10))
        rows = rec[rmask != 0] if masked else rec
        r = min(len(sel), len(rows))
        slots, cnt = s.update_distinct(p, dev, torch.from_numpy(rmask).cuda() if masked else None, op=op)
        assert int(cnt) == r
        np.testing.assert_array_equal(np_of(slots)[:r], sel[:r])
        for f in range(F):
            fld[f][sel[:r]] = rows[:r, f] + (fld[f][sel[:r]] if op == abm.OP_ADD else 0)
        check(f"update {masked}")
    m = torch.from_numpy((rng.random(n + 1) < 0.3).astype(np.int32)).cuda()[1:]  # not 16-byte aligned
    gone = (act != 0) & (np_of(m) != 0)
    assert int(s.remove(abm.pred(abm.PRED_MASK, mask=m))) == int(gone.sum())
    act[gone] = 0
    check("remove")
    for id_field in (-1, F - 1):
        free = np.flatnonzero(act == 0)
        r = min(k, len(free))
        first = s.counters()["next_id"]
        slots, cnt = s.add(dev, id_field=id_field)
        assert int(cnt) == r
        np.testing.assert_array_equal(np_of(slots)[:r], free[:r])
        act[free[:r]] = 1
        for f in range(F):
            fld[f][free[:r]] = first + np.arange(r) if f == id_field else rec[:r, f]
        check(f"add {id_field}")
    # the fused call against remove, update and add of the oracle's draws
    o = oracle.Slab(n, F)
    o.active[:] = np_of(s.read(-1))
    for f in range(F):
        o.fields[f][:] = fld[f]
    if F <= 8:
        T, kk = workloads.threshold(0.3), max(1, n // 5)
        a = s.philox_records(4, abm.P_NEWREC0, abm.P_NEWREC1, kk)
        b = s.philox_records(4, abm.P_DELTA0, abm.P_DELTA1, kk)
        s.selective_update(4, T, a, b)
        o.c1_call(4, T, kk, seed=9)
        np.testing.assert_array_equal(np_of(s.read(-1)) != 0, o.active != 0)
        for f in range(F):
            np.testing.assert_array_equal(np_of(s.read(f)), o.fields[f])
    s.check()


@pytest.mark.parametrize("n,p", [(262_145, 0.015), (300_001, 0.017), (300_001, 0.05), (300_001, 0.5),
                                 (2_000_003, 0.02), (2_000_003, 0.3)])
def test_selective_update_paths(eng, n, p):
    """Whole numbers, so exact: the two sides of the record-moving line, from a half-full set on, with flags other
    than 0 and 1: those are rewritten as 1 exactly in the 16-slot groups that receive an agent and the 8-slot groups
    that lose one."""
    from paper_2508_16508_gb300 import abm
    T, k = workloads.threshold(p), workloads.k_for(p, n)
    s, o = eng.Slab(n, 8, seed=2, init=abm.INIT_HALF_LIVE), oracle.Slab(n, 8)
    o.c1_init(seed=2)
    odd = np.where(o.active & (np.arange(n) % 37 == 0), 5, o.active).astype(np.int32)
    s.write(-1, torch.from_numpy(odd).cuda())
    for step in range(4):
        rec = s.philox_records(step, abm.P_NEWREC0, abm.P_NEWREC1, k)
        dl = s.philox_records(step, abm.P_DELTA0, abm.P_DELTA1, k)
        before, ids = o.active.copy(), o.fields.copy()
        s.selective_update(step, T, rec, dl)
        o.c1_call(step, T, k, seed=2)
        draws = np.zeros(-(-n // 16) * 16, bool)
        new = draws.copy()
        new[:n] = (o.fields != ids).any(0) & (o.active != 0)  # added or updated
        got = np_of(s.read(-1))
        np.testing.assert_array_equal(got != 0, o.active != 0)
        for f in range(8):
            np.testing.assert_array_equal(np_of(s.read(f)), o.fields[f])
        # a flag that keeps an odd value was live, stays live, and lies in no group that was written
        np.testing.assert_array_equal(got[got > 1], odd[got > 1])
        freed = np.zeros_like(new)
        freed[:n] = (before != 0) & (o.active == 0)  # certainly removed
        wrote = np.repeat(freed.reshape(-1, 8).any(1), 8)[:n]
        filled = np.zeros_like(new)
        filled[:n] = (before == 0) & (o.active != 0)  # certainly added
        wrote |= np.repeat(filled.reshape(-1, 16).any(1), 16)[:n]
        assert got[wrote].max(initial=0) <= 1
        odd = got
    s.check()


@pytest.mark.parametrize("n,p", [(2_000_003, 0.0038), (2_000_003, 0.0041), (300_001, 0.001), (300_001, 0.01)])
def test_selective_update_early_and_late_flags(eng, n, p):
    """The same on both sides of the number of records from which removed slots' flags are written late."""
    test_selective_update_paths(eng, n, p)


@pytest.mark.parametrize("n,p", [(300_001, 0.02), (270_003, 0.06)])
def test_selective_update_while_the_set_fills(eng, n, p):
    """From a half-full set to a full one and, emptied, on again: the launches change on the way (whole numbers, so
    exact). With and without waiting for a call before the next is made."""
    from paper_2508_16508_gb300 import abm
    T, k = workloads.threshold(p), workloads.k_for(p, n)
    s, o = eng.Slab(n, 8, seed=6, init=abm.INIT_HALF_LIVE), oracle.Slab(n, 8)
    o.c1_init(seed=6)
    for step in range(int(8 / p)):
        if step == int(5 / p):
            keep = (np.arange(n) % 3 == 0).astype(np.int32)
            s.remove(abm.pred(abm.PRED_MASK, mask=torch.from_numpy(1 - keep).cuda()))
            o.active[:] = o.active * keep
        c = s.selective_update(step, T, s.philox_records(step, abm.P_NEWREC0, abm.P_NEWREC1, k),
                               s.philox_records(step, abm.P_DELTA0, abm.P_DELTA1, k))
        d = o.c1_call(step, T, k, seed=6)
        if step % 3 == 0:
            assert np_of(c).tolist() == [d["removed"], d["added"], d["updated"]]
    np.testing.assert_array_equal(np_of(s.read(-1)), o.active)
    for f in range(8):
        np.testing.assert_array_equal(np_of(s.read(f)), o.fields[f])
    assert s.counters()["n_active"] == int(o.active.sum())
    s.check()


@pytest.mark.parametrize("n,p", [(2_400_003, 0.06)])
def test_selective_update_fills_the_second_wave(eng, n, p):
    """The same in sets whose ranking pass takes more than one wave of CTAs."""
    test_selective_update_while_the_set_fills(eng, n, p)


@pytest.mark.parametrize("threads,ctas", [(128, 16), (256, 2), (512, 4)])
@pytest.mark.parametrize("F,p", [(8, 0.002), (8, 0.008), (8, 0.1), (5, 0.002), (5, 0.008), (5, 0.1)])
def test_selective_update_shapes(eng, threads, ctas, F, p):
    """Every launch shape of the passes takes each of their ways (whole numbers, so exact)."""
    n = 700_001
    T, k = workloads.threshold(p), workloads.k_for(p, n)
    s, o = eng.Slab(n, F, seed=3, init=1), oracle.Slab(n, F)
    s.tune(threads, ctas)
    o.c1_init(seed=3)
    from paper_2508_16508_gb300 import abm
    for step in range(6):
        s.selective_update(step, T, s.philox_records(step, abm.P_NEWREC0, abm.P_NEWREC1, k),
                           s.philox_records(step, abm.P_DELTA0, abm.P_DELTA1, k))
        o.c1_call(step, T, k, seed=3)
    np.testing.assert_array_equal(np_of(s.read(-1)), o.active)
    for f in range(F):
        np.testing.assert_array_equal(np_of(s.read(f)), o.fields[f])
    s.check()


@pytest.mark.parametrize("M,R,levels", [(4095, 3, 1), (4097, 70_000, 2), (700_003, 5, 1), (700_003, 50_000, 3),
                                        (1_500_000, 1, 2**32), (1_300_001, 1_000_000, 2**32)])
def test_resolve_ties_and_hot_resources(eng, M, R, levels):
    """Whole numbers, so exact: few priority levels (ties go to the smaller index, across chunks and CTAs) and
    resources claimed by a large share of all, at the sizes around the kernel's chunks; top priorities and resources."""
    rng = np.random.default_rng(M + R)
    res = np.where(rng.random(M) < 0.3, R - 1, rng.integers(0, R, M)).astype(np.int32)
    prio = rng.integers(0, levels, M).astype(np.uint32)
    prio[rng.random(M) < 0.1] = 0xFFFFFFFF
    order = np.lexsort((np.arange(M), prio, res))
    first = order[np.r_[True, res[order][1:] != res[order][:-1]]]
    want = np.full(R, -1, np.int64)
    want[res[first]] = first
    won = np.zeros(M, np.uint8)
    won[first] = 1
    r = eng.Resolver(R)
    isw = torch.empty(M, dtype=torch.uint8, device="cuda")
    w = r(torch.from_numpy(res).cuda(), torch.from_numpy(prio.view(np.int32)).cuda(), isw)
    np.testing.assert_array_equal(np_of(w), want)
    np.testing.assert_array_equal(np_of(isw), won)
    assert torch.all(r.table == -1)


def same_place(first, count, R):
    """Resources of one place of k_claims' shared table, `first` among them: 13 bits of a product."""
    place = ((np.arange(R, dtype=np.uint64) * 2654435761) & 0xFFFFFFFF) >> 19
    return np.nonzero(place == place[first])[0][:count].astype(np.int32)


@pytest.mark.parametrize("M", [1, 1023, 1025, 4097, 50_000, 2_000_003])
@pytest.mark.parametrize("first,count,crowd", [(0, 2, 0.0), (0, 5, 0.3), (5, 3, 0.9), (777, 31, 0.0)])
def test_resolve_resources_that_share_a_place(eng, M, first, count, crowd):
    """Whole numbers, so exact: hot resources that all have the same first place of the shared table, alone and among
    claims on all others, with ties and claims outside the range."""
    R = 1 << 18
    rng = np.random.default_rng(M + count)
    hot = same_place(first, count, R)
    assert len(hot) == count
    res = np.where(rng.random(M) < crowd, rng.integers(-2, R + 2, M), hot[rng.integers(0, count, M)]).astype(np.int32)
    prio = rng.integers(0, 1000, M).astype(np.uint32)
    r = eng.Resolver(R)
    isw = torch.empty(M, dtype=torch.uint8, device="cuda")
    w = r(torch.from_numpy(res).cuda(), torch.from_numpy(prio.view(np.int32)).cuda(), isw)
    ow, oisw = oracle.resolve(res, prio, R)
    np.testing.assert_array_equal(np_of(w), ow)
    np.testing.assert_array_equal(np_of(isw), oisw)
    assert torch.all(r.table == -1)


@pytest.mark.parametrize("F,shift", [(1, 0), (2, 1), (4, 0), (5, 0), (8, 1), (8, 4), (11, 3), (12, 0), (12, 2), (13, 0),
                                     (16, 4), (16, 1)])
def test_row_shapes(eng, F, shift):
    """Whole numbers, so exact: rows of every width and records at every alignment above the one-launch sizes."""
    from paper_2508_16508_gb300 import abm
    n, k = 262_150, 40_003
    rng = np.random.default_rng(F * 8 + shift)
    s = eng.Slab(n, F, seed=9)
    act = (rng.random(n) < 0.5).astype(np.int32)
    fld = rng.integers(-50, 50, (F, n)).astype(np.int32)
    s.write(-1, torch.from_numpy(act).cuda())
    for f in range(F):
        s.write(f, torch.from_numpy(fld[f]).cuda())
    rec = rng.integers(-2**31, 2**31, (k, F)).astype(np.int32)
    rmask = (rng.random(k) < 0.5).astype(np.int32)
    dev = torch.zeros(k * F + shift, dtype=torch.int32, device="cuda")[shift:].view(k, F)
    dev.copy_(torch.from_numpy(rec))
    for mask, op in ((None, abm.OP_ADD), (None, abm.OP_SET), (rmask, abm.OP_ADD), (rmask, abm.OP_SET)):
        sel = np.flatnonzero((act != 0) & (fld[0] >= -10))
        rows = rec if mask is None else rec[mask != 0]
        r = min(len(sel), len(rows))
        s.update_distinct(abm.pred(abm.PRED_FIELD, field=0, cmp=abm.CMP_GE, value=-10), dev,
                          None if mask is None else torch.from_numpy(mask).cuda(), op=op)
        for f in range(F):
            fld[f][sel[:r]] = rows[:r, f] + (fld[f][sel[:r]] if op == abm.OP_ADD else 0)
    for id_field in (-1, 0, F - 1):
        free = np.flatnonzero(act == 0)[:k]
        first = s.counters()["next_id"]
        s.add(dev, id_field=id_field)
        for f in range(F):
            fld[f][free] = rec[:len(free), f] if f != id_field else first + np.arange(len(free))
        act[free] = 1
    for f in range(F):
        np.testing.assert_array_equal(np_of(s.read(f)), fld[f], err_msg=str(f))
    np.testing.assert_array_equal(np_of(s.read(-1)) != 0, act != 0)
    s.check()


@pytest.mark.parametrize("F", [1, 4, 5, 7])
def test_selective_update_row_shapes(eng, F):
    """The same for the one call of the three operations, against the oracle."""
    from paper_2508_16508_gb300 import abm
    n, p = 270_001, 0.2
    T, k = workloads.threshold(p), workloads.k_for(p, n)
    s, o = eng.Slab(n, F, seed=4, init=abm.INIT_HALF_LIVE), oracle.Slab(n, F)
    o.c1_init(seed=4)
    for step in range(3):
        s.selective_update(step, T, s.philox_records(step, abm.P_NEWREC0, abm.P_NEWREC1, k),
                           s.philox_records(step, abm.P_DELTA0, abm.P_DELTA1, k))
        o.c1_call(step, T, k, seed=4)
    np.testing.assert_array_equal(np_of(s.read(-1)) != 0, o.active != 0)
    for f in range(F):
        np.testing.assert_array_equal(np_of(s.read(f)), o.fields[f])
    s.check()


@pytest.mark.parametrize("n,F,k,shift", [(262_144, 4, 31_000, 0), (262_144, 4, 33_000, 0), (131_072, 11, 46_000, 0),
                                         (131_072, 11, 48_000, 0), (262_144, 8, 4500, 0), (262_144, 8, 4800, 1),
                                         (262_144, 16, 300, 1), (200_001, 1, 28_000, 0), (200_001, 5, 10_000, 0),
                                         (131_073, 8, 200_000, 0), (131_000, 8, 131_000, 0), (100_003, 13, 90_000, 3),
                                         (100_003, 3, 9_000, 0), (65_536, 15, 70_000, 0), (60_000, 15, 3000, 0),
                                         (1025, 7, 1025, 0), (5, 12, 9, 2)])
def test_record_moves_of_small_sets(eng, n, F, k, shift):
    """Whole numbers, so exact: sets of up to 262,144 slots on both sides of the number of records above which the calls
    take the passes, and of that above which a cluster splits crowded records evenly; records at every alignment, every
    id field, some flags odd."""
    from paper_2508_16508_gb300 import abm
    rng = np.random.default_rng(n + F + k)
    s = eng.Slab(n, F, seed=9)
    act = np.where(rng.random(n) < 0.5, rng.choice([1, 1, 1, 7], n), 0).astype(np.int32)
    fld = rng.integers(-50, 50, (F, n)).astype(np.int32)
    s.write(-1, torch.from_numpy(act).cuda())
    for f in range(F):
        s.write(f, torch.from_numpy(fld[f]).cuda())
    rec = rng.integers(-2**31, 2**31, (k, F)).astype(np.int32)
    dev = torch.zeros(k * F + shift, dtype=torch.int32, device="cuda")[shift:].view(k, F)
    dev.copy_(torch.from_numpy(rec))
    rmask = (rng.random(min(k, n)) < 0.5).astype(np.int32)

    def check(where):
        for f in range(F):
            np.testing.assert_array_equal(np_of(s.read(f)), fld[f], err_msg=f"{where}, field {f}")
        np.testing.assert_array_equal(np_of(s.read(-1)) != 0, act != 0, err_msg=where)

    for masked, op in ((False, abm.OP_ADD), (False, abm.OP_SET), (True, abm.OP_ADD), (True, abm.OP_SET)):
        sel = np.flatnonzero((act != 0) & (fld[0] >= -30))
        rows = rec[:len(rmask)][rmask != 0] if masked else rec
        r = min(len(sel), len(rows))
        slots, cnt = s.update_distinct(abm.pred(abm.PRED_FIELD, field=0, cmp=abm.CMP_GE, value=-30),
                                       dev[:len(rmask)] if masked else dev,
                                       torch.from_numpy(rmask).cuda() if masked else None, op=op)
        assert int(cnt) == r
        np.testing.assert_array_equal(np_of(slots)[:r], sel[:r])
        for f in range(F):
            fld[f][sel[:r]] = rows[:r, f] + (fld[f][sel[:r]] if op == abm.OP_ADD else 0)
        check(f"update {masked} {op}")
    for id_field in [-1] + list(range(F)):
        gone = rng.random(n) < 0.4
        s.remove(abm.pred(abm.PRED_MASK, mask=torch.from_numpy(gone.astype(np.int32)).cuda()))
        act[gone] = 0
        free = np.flatnonzero(act == 0)
        r = min(k, len(free))
        first = s.counters()["next_id"]
        slots, cnt = s.add(dev, id_field=id_field)
        assert int(cnt) == r
        np.testing.assert_array_equal(np_of(slots)[:r], free[:r])
        act[free[:r]] = 1
        for f in range(F):
            fld[f][free[:r]] = first + np.arange(r) if f == id_field else rec[:r, f]
        check(f"add {id_field}")
    if F <= 8:
        o = oracle.Slab(n, F)
        o.active[:] = np_of(s.read(-1))
        for f in range(F):
            o.fields[f][:] = fld[f]
        for step in range(2):
            s.selective_update(step, workloads.threshold(0.3), s.philox_records(step, abm.P_NEWREC0, abm.P_NEWREC1, k),
                               s.philox_records(step, abm.P_DELTA0, abm.P_DELTA1, k))
            o.c1_call(step, workloads.threshold(0.3), k, seed=9)
        np.testing.assert_array_equal(np_of(s.read(-1)) != 0, o.active != 0)
        for f in range(F):
            np.testing.assert_array_equal(np_of(s.read(f)), o.fields[f])
    s.check()
