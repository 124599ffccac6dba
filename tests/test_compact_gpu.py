"""Compact streams (scalar and data-axis tapes) against the general interpreter.

A tape built with NDVM_COMPACT=0 runs on the general kernels.  Both run the same plan; they
differ in the order in which a data sum's points are added (points per thread) and in
roundings of the reverse rules that the compact form fuses, so lanes agree within the parity bound
(1e-12 in binary64, 1e-5 in binary32, of the lane's largest component; more only where the oracle's two
derivative engines disagree by more, as in the parity tests).  Sizes cover the edges of the split:
fewer points than threads, one more or less than a pass, one lane, ragged warps."""
import numpy as np
import pytest

import workloads as W
from conftest import oracle_ref, rel_check

pytestmark = pytest.mark.gpu

BODY = ("(model (params a b c) (+ (* 0.5 (sin a)) (/ (exp b) (+ 1.0 (* c c)))\n"
        "  (data-sum {n} 2 (let* ((x (dobs 0)) (u (* a x)) (v (/ u (+ 1.0 (* b b x x))))\n"
        "    (w (if (< u c) (tanh v) (log (+ 1.5 (* v v))))) (r (- (+ w (pow u 3) (sqrt (+ 1.0 (* v v))) (abs v)) (dobs 1))))\n"
        "    (* r r)))\n"
        "  (data-sum 3 1 (* c (dobs 0)))))")


def _both(ndvm, w, dtype, monkeypatch):
    import torch
    fast = ndvm.trace_build(w.program, w.frontend)
    monkeypatch.setenv("NDVM_COMPACT", "0")
    general = ndvm.trace_build(w.program, w.frontend)
    monkeypatch.delenv("NDVM_COMPACT")
    p = torch.tensor(w.params, dtype=dtype, device="cuda")
    o = torch.tensor(w.obs, dtype=dtype, device="cuda")
    out = [ndvm.value_and_grad(t, p, o) + (ndvm.forward(t, p, o),) for t in (fast, general)]
    torch.cuda.synchronize()
    for t in (fast, general):
        ndvm.check_device(t)
    return [[x.cpu().numpy().astype(np.float64) for x in r] for r in out]


@pytest.mark.parametrize("dtype", ["float64", "float32"])
@pytest.mark.parametrize("B,n", [(1, 0), (1, 1), (2, 2), (31, 31), (33, 32), (64, 33), (5, 63), (7, 64), (3, 65), (40, 129),
                                 (1, 1000), (700, 257), (5000, 5), (20000, 3), (30001, 2), (30001, 7)])
def test_compact_equals_general(ndvm, oracle_mod, cuda, monkeypatch, B, n, dtype):
    import torch
    rng = np.random.default_rng(B + n)
    w = W.Workload("body", BODY.format(n=n), 0, rng.normal(size=(B, 3)), rng.normal(size=max(2 * n, 3)), np.zeros(3))
    f64 = dtype == "float64"
    fast, general = _both(ndvm, w, getattr(torch, dtype), monkeypatch)
    idx = np.unique([0, B // 2, B - 1])
    ok, rep = rel_check(fast[0], fast[1], general[0], general[1], 1e-12 if f64 else 1e-5)
    assert ok, rep
    np.testing.assert_array_equal(fast[0], fast[2])  # the value plan's loss is the gradient plan's
    if f64:
        ol, og, sp = oracle_ref(oracle_mod, w.program, w.params[idx], w.obs)
        ok, rep = rel_check(fast[0][idx], fast[1][idx], ol, og, 1e-12, sp)
        assert ok, rep


@pytest.mark.parametrize("steps", [3, 700])
def test_no_points_beside_a_long_stream(ndvm, cuda, monkeypatch, steps):
    """A data sum over no points in a stream of more records than shared memory holds."""
    import torch
    rng = np.random.default_rng(steps)
    text = ("(model (params a b) (+ (data-sum 0 1 (* a (dobs 0)))"
            f" (let loop ((i 0) (x a)) (if (= i {steps}) x (loop (+ i 1) (+ (* x b) (sin x)))))))")
    w = W.Workload("no_points", text, 0, rng.uniform(-0.5, 0.5, (70, 2)), np.zeros(1), np.zeros(2))
    fast, general = _both(ndvm, w, torch.float64, monkeypatch)
    ok, rep = rel_check(fast[0], fast[1], general[0], general[1], 1e-12)
    assert ok, rep
    np.testing.assert_array_equal(fast[0], fast[2])


@pytest.mark.parametrize("dtype", ["float64", "float32"])
@pytest.mark.parametrize("terms,values", [(20, 1), (165, 1), (20, 70), (20, 75)])
def test_value_and_gradient_plans_add_in_the_same_order(ndvm, cuda, terms, values, dtype):
    """The second and the last body's gradient stream alone is too long for the compact form: the value
    plan then runs on the general kernel as well, and the loss keeps its bits."""
    import torch
    rng = np.random.default_rng(terms)
    u = " ".join(f"(v{i} (sin (* {0.1 + 0.01 * i} (* b x))))" for i in range(values))
    t = " ".join(f"(* v{i % values} (+ a (* {0.5 + i} x)))" for i in range(max(terms, values)))
    text = (f"(model (params a b) (data-sum 301 2 (let* ((x (dobs 0)) {u} (r (- (+ {t}) (dobs 1)))) (* r r))))")
    tape = ndvm.trace_build(text)
    p = torch.tensor(rng.normal(size=(300, 2)), dtype=getattr(torch, dtype), device=cuda)
    o = torch.tensor(rng.normal(size=602), dtype=getattr(torch, dtype), device=cuda)
    loss, _ = ndvm.value_and_grad(tape, p, o)
    np.testing.assert_array_equal(ndvm.forward(tape, p, o).cpu().numpy(), loss.cpu().numpy())


def _special():
    """Lanes of zeros, infinities, NaN, subnormals and the largest values through every scalar rule."""
    s = np.array([0.0, -0.0, 1.0, -1.0, np.inf, -np.inf, np.nan, 5e-324, -1e-310, 1e-8, 1.7e308, -3.0, 709.0, 1e6])
    a, b, c = np.meshgrid(s, s, s)
    return np.stack([a.ravel(), b.ravel(), c.ravel()], 1)


@pytest.mark.parametrize("n", [1, 40])
def test_compact_special_values(ndvm, cuda, monkeypatch, n):
    """Non-finite lanes keep their class and finite ones their values (the same rules run on the same operands)."""
    import torch
    rng = np.random.default_rng(n)
    obs = rng.normal(size=max(2 * n, 3))
    w = W.Workload("special", BODY.format(n=n), 0, _special(), obs, np.zeros(3))
    fast, general = _both(ndvm, w, torch.float64, monkeypatch)
    for f, g in zip(fast, general):
        assert np.array_equal(np.isnan(f), np.isnan(g)) and np.array_equal(np.isposinf(f), np.isposinf(g))
        assert np.array_equal(np.isneginf(f), np.isneginf(g))
        fin = np.isfinite(g)
        # sums of magnitudes up to 1e308 in another order: bounded by their size, lane by lane
        np.testing.assert_allclose(f[fin], g[fin], rtol=1e-9, atol=1e-300)


@pytest.mark.parametrize("dtype", ["float64", "float32"])
@pytest.mark.parametrize("make", [
    lambda: W.logistic(B=1, n_obs=3, every=2), lambda: W.logistic(B=1000, n_obs=7, every=13),
    lambda: W.logistic(B=130, n_obs=100, every=10), *[lambda k=k: W.second_client(B=65)[k] for k in range(4)],
    *[lambda k=k: W.control_fuzz(12, B=70, n_points=19, seed=5)[k] for k in range(12)],
    *[lambda k=k: W.random_exprs(8, B=150, n_points=50, seed=3)[k] for k in range(8)]])
def test_compact_programs(ndvm, oracle_mod, cuda, monkeypatch, make, dtype):
    import torch
    w = make()
    fast, general = _both(ndvm, w, getattr(torch, dtype), monkeypatch)
    f64 = dtype == "float64"
    _, _, spread = oracle_ref(oracle_mod, w.program, w.params, w.obs, frontend=w.frontend, f32=not f64)
    ok, rep = rel_check(fast[0], fast[1], general[0], general[1], 1e-12 if f64 else 1e-5, spread)
    assert ok, rep


@pytest.mark.parametrize("dtype", ["float64", "float32"])
@pytest.mark.parametrize("lanes", [[300] * 14, [2000, 1, 900, 4000, 33] * 2, [20000, 15000, 40]])
def test_batches_past_the_resident_blocks(ndvm, cuda, lanes, dtype):
    """Members share a launch of more blocks than the GPU holds at once, ordered by length: the same
    bits as separate calls."""
    import torch
    ws = W.random_exprs(len(lanes), B=2, n_points=70, seed=99)
    tapes = [ndvm.trace_build(w.program, w.frontend) for w in ws]
    dt = getattr(torch, dtype)
    params = [torch.tensor(w.params[:1].repeat(n, 0) + 1e-4 * np.arange(n)[:, None], dtype=dt, device=cuda)
              for w, n in zip(ws, lanes)]
    obs = [torch.tensor(w.obs, dtype=dt, device=cuda) for w in ws]
    loss, grad = ndvm.value_and_grad_multi(tapes, params, obs)
    for t, p, o, l, g in zip(tapes, params, obs, loss, grad):
        l1, g1 = ndvm.value_and_grad(t, p, o)
        np.testing.assert_array_equal(l.cpu().numpy(), l1.cpu().numpy())
        np.testing.assert_array_equal(g.cpu().numpy(), g1.cpu().numpy())
