"""GPU parity of the capacity predictor's kernels vs the float64 reference,
and bit-exactness of learned-capacity batching vs fixed capacity."""
import os

import numpy as np
import pytest

import workloads
from oracle import mlp as omlp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

WEIGHTS = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                       "paper_2508_16508_gb300", "data", "capacity_mlp.npz")


@pytest.fixture(scope="module")
def cap():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2508_16508_gb300 import abm, capacity
    abm.lib()
    return capacity


def dims_of(m):
    return [12] + [m.hidden] * m.layers + [2]


@pytest.mark.parametrize("hidden,layers,B", [(128, 3, 300), (32, 2, 1000), (128, 3, 4099)])
def test_gradients_vs_float64(cap, hidden, layers, B):
    rng = np.random.default_rng(B)
    m = cap.CapacityModel(workloads.predation_params(), hidden=hidden, layers=layers, seed=B)
    x = rng.normal(size=(B, 12)).astype(np.float32)
    y = rng.normal(size=(B, 2)).astype(np.float32) * 2
    xd, yd = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    loss = m.gradients(xd, yd, tau=0.99)
    g = m.grads().cpu().numpy().astype(np.float64)
    p = m.params().cpu().numpy()
    layers64 = omlp.unflatten(p, dims_of(m))
    ol, og = omlp.loss_and_grads(layers64, x.astype(np.float64), y.astype(np.float64), 0.99)
    og = omlp.flatten(og)
    assert abs(float(loss.item()) - ol) <= 1e-4 * abs(ol) + 1e-6
    scale = np.abs(og).max()
    np.testing.assert_allclose(g, og, rtol=1e-4, atol=1e-4 * scale)
    # forward
    yh = m.predict(xd).cpu().numpy()
    np.testing.assert_allclose(yh, omlp.forward(layers64, x.astype(np.float64))[-1], rtol=1e-4,
                               atol=1e-4 * np.abs(yh).max())


def test_gradients_with_row_permutation(cap):
    rng = np.random.default_rng(7)
    N, B = 5000, 1024
    m = cap.CapacityModel(workloads.predation_params(), seed=3)
    x = rng.normal(size=(N, 12)).astype(np.float32)
    y = rng.normal(size=(N, 2)).astype(np.float32)
    a, c, m0 = 3001, 17, 2048
    rows = (a * (m0 + np.arange(B)) + c) % N
    m.gradients(torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda(), tau=0.99, B=B, perm=(N, a, c, m0))
    g = m.grads().cpu().numpy()
    layers64 = omlp.unflatten(m.params().cpu().numpy(), dims_of(m))
    _, og = omlp.loss_and_grads(layers64, x[rows].astype(np.float64), y[rows].astype(np.float64), 0.99)
    og = omlp.flatten(og)
    np.testing.assert_allclose(g, og, rtol=1e-4, atol=1e-4 * np.abs(og).max())


def test_adam_step_vs_float64(cap):
    rng = np.random.default_rng(1)
    m = cap.CapacityModel(workloads.predation_params(), hidden=32, layers=2, seed=5)
    x = torch.from_numpy(rng.normal(size=(512, 12)).astype(np.float32)).cuda()
    y = torch.from_numpy(rng.normal(size=(512, 2)).astype(np.float32)).cuda()
    p = m.params().cpu().numpy().astype(np.float64)
    mom, vel = np.zeros_like(p), np.zeros_like(p)
    for t in range(1, 4):
        m.gradients(x, y)
        g = m.grads().cpu().numpy().astype(np.float64)
        m.train_step(x, y, lr=1e-2)
        p, mom, vel = omlp.adam_step(p, g, mom, vel, t, lr=1e-2)
        np.testing.assert_allclose(m.params().cpu().numpy(), p, rtol=2e-5, atol=2e-6)


def test_features_and_capacity(cap):
    tab = workloads.sample_models(300, 5)
    models = [dict(side=int(tab["side"][i]), n0=tab["n0"][i], params=tab["params"][i]) for i in range(300)]
    m = cap.CapacityModel(workloads.predation_params())
    table = cap.table_of(models, 500)
    x = m.features(table).cpu().numpy()
    np.testing.assert_allclose(x, omlp.features(table, workloads.predation_params()), rtol=1e-6, atol=1e-6)
    yh = np.random.default_rng(0).normal(size=(300, 2)).astype(np.float32) * 3 + 6
    caps_max = workloads.fixed_caps(tab["side"])
    got = None
    import ctypes as C
    from paper_2508_16508_gb300 import abm
    yd = torch.from_numpy(yh).cuda()
    cm = torch.from_numpy(caps_max).cuda()
    n0 = torch.from_numpy(tab["n0"]).cuda()
    out = torch.empty_like(cm)
    abm.call("abm_capacity_from_prediction", abm.ptr(yd), 300, 0.1, 128, abm.ptr(cm), abm.ptr(n0), abm.ptr(out),
             abm.stream_handle())
    got = out.cpu().numpy()
    want = omlp.capacity(yh.astype(np.float64), 0.1, 128, caps_max, tab["n0"])
    assert np.mean(got == want) > 0.999 and np.abs(got - want).max() <= 128


def test_training_reduces_loss_and_hits_quantile(cap):
    rng = np.random.default_rng(2)
    N = 8192
    x = rng.normal(size=(N, 12)).astype(np.float32)
    # target: a smooth function plus noise; the 0.99 quantile sits ~2.33 sd above it
    y = (np.stack([x[:, 0] * 0.5 + x[:, 1], x[:, 2] - x[:, 3] * 0.3], 1) +
         0.2 * rng.normal(size=(N, 2))).astype(np.float32)
    m = cap.CapacityModel(workloads.predation_params(), seed=1)
    xd, yd = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    l0 = float(m.gradients(xd, yd).item())
    m.fit(xd, yd, epochs=60, batch=512, lr=2e-3)
    l1 = float(m.gradients(xd, yd).item())
    assert l1 < 0.2 * l0
    cover = np.mean(y <= m.predict(xd).cpu().numpy())
    assert 0.95 < cover <= 1.0


def test_learned_capacity_is_bit_exact(cap):
    """Tight (deliberately too small for some) capacities + device overflow
    detection + fixed-capacity rerun == the fixed-capacity run, model by model."""
    from paper_2508_16508_gb300 import engine
    tab = workloads.sample_models(384, 21, side_lo=16, side_hi=64)
    fixed = workloads.fixed_caps(tab["side"])
    models = [dict(side=int(tab["side"][i]), seed=9, model=i, params=tab["params"][i], cap=fixed[i],
                   n0=tab["n0"][i]) for i in range(384)]
    b = engine.Batch(models)
    b.run(80)
    want = b.digest().cpu().numpy()
    want_cnt = b.counters()
    del b
    hw = np.array([c["hw"] for c in want_cnt])
    rng = np.random.default_rng(0)
    learned = np.maximum(np.ceil(hw * rng.uniform(0.8, 1.6, size=hw.shape)), tab["n0"]).astype(np.int32)
    res = cap.run_learned(models, learned, fixed, 80)
    assert len(res["overflowed"]) > 0
    np.testing.assert_array_equal(res["digest"], want)
    for got, w in zip(res["counters"], want_cnt):
        assert got["n_active"] == w["n_active"] and got["hw"] == w["hw"] and got["next_id"] == w["next_id"]


@pytest.mark.skipif(not os.path.exists(WEIGHTS), reason="trained weights not present")
def test_trained_predictor_gain(cap):
    """What the trained network buys: on models of the batched workload's
    sampler (seed disjoint from training), far less capacity than the fixed
    worst case, few overflows, and results equal to the fixed-capacity run."""
    from paper_2508_16508_gb300 import engine
    n, steps = 512, 200
    tab = workloads.sample_models(n, workloads.BATCH["sampler_seed"])
    fixed = workloads.fixed_caps(tab["side"])
    models = [dict(side=int(tab["side"][i]), seed=workloads.BATCH["philox_seed"], model=i,
                   params=tab["params"][i], cap=fixed[i], n0=tab["n0"][i]) for i in range(n)]
    m = cap.CapacityModel.load(WEIGHTS)
    learned = m.capacities(m.features(cap.table_of(models, steps)), fixed, tab["n0"])
    b = engine.Batch(models)
    b.run(steps)
    want = b.digest().cpu().numpy()
    del b
    res = cap.run_learned(models, learned, fixed, steps)
    np.testing.assert_array_equal(res["digest"], want)
    assert learned.sum() < 0.5 * fixed.sum()
    assert len(res["overflowed"]) <= 0.05 * n


@pytest.mark.parametrize("n_in,hidden,layers,n_out,B", [
    (12, 128, 3, 2, 1), (12, 37, 1, 2, 7), (1, 100, 2, 1, 9), (128, 64, 8, 8, 129), (12, 128, 3, 2, 2433),
    (13, 127, 2, 5, 5001), (12, 128, 4, 2, 300), (12, 130, 2, 2, 77), (12, 64, 2, 9, 260)])
def test_net_shapes_vs_float64(cap, n_in, hidden, layers, n_out, B):
    """Both training paths (weights resident in shared memory; one GEMM per product) at the edges of their slabs,
    tiles and widths: gradients, forward and loss. Tolerance: float32 sums of up to 5001 x 128 terms, 1e-4 of the
    largest entry."""
    import ctypes as C
    from paper_2508_16508_gb300 import abm
    rng = np.random.default_rng(B)
    h = C.c_void_p()
    abm.call("abm_mlp_create", n_in, hidden, layers, n_out, 3, B, abm.stream_handle(), C.byref(h))
    try:
        cnt = C.c_int64()
        abm.call("abm_mlp_params", h, None, None, C.byref(cnt))
        dims = [n_in] + [hidden] * layers + [n_out]
        p = (rng.normal(size=cnt.value) * (2.0 / hidden) ** 0.5).astype(np.float32)  # biases too
        x = rng.normal(size=(B, n_in)).astype(np.float32)
        y = rng.normal(size=(B, n_out)).astype(np.float32) * 2
        pd, xd, yd = (torch.from_numpy(v).cuda() for v in (p, x, y))
        abm.call("abm_mlp_set_params", h, abm.ptr(pd), cnt.value, abm.stream_handle())
        out, loss, g = torch.empty(B, n_out).cuda(), torch.zeros(1).cuda(), torch.empty(cnt.value).cuda()
        abm.call("abm_mlp_forward", h, abm.ptr(xd), B, abm.ptr(out), abm.stream_handle())
        abm.call("abm_mlp_gradients", h, abm.ptr(xd), abm.ptr(yd), B, 0.9, 0, 0, 0, 0, abm.ptr(loss),
                 abm.stream_handle())
        abm.call("abm_mlp_get_grads", h, abm.ptr(g), cnt.value, abm.stream_handle())
        torch.cuda.synchronize()
        net = omlp.unflatten(p, dims)
        ref = omlp.forward(net, x.astype(np.float64))[-1]
        ol, og = omlp.loss_and_grads(net, x.astype(np.float64), y.astype(np.float64), 0.9)
        og = omlp.flatten(og)
        np.testing.assert_allclose(out.cpu().numpy(), ref, rtol=1e-4, atol=1e-4 * np.abs(ref).max())
        np.testing.assert_allclose(g.cpu().numpy(), og, rtol=1e-4, atol=1e-4 * np.abs(og).max())
        assert abs(float(loss.item()) - ol) <= 1e-4 * abs(ol) + 1e-6
    finally:
        abm.call("abm_mlp_destroy", h)
