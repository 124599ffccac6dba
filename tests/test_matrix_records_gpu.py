"""Matrix records (tapes with matrices and no data axis) against the general interpreter.

A tape built with NDVM_COMPACT=0 runs on the general kernels.  Both run the same plan with the
same sums in the same order, except that a product with a constant matrix leaves out the terms of its
zeros (which add nothing): on these programs the results are equal bit for bit, but for the sign of a
zero.  Non-finite lanes take every term: they keep their class."""
import numpy as np
import pytest

import workloads as W
from conftest import matrix_program, oracle_ref, rel_check

pytestmark = pytest.mark.gpu


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
@pytest.mark.parametrize("make", [
    *[lambda B=B, T=T: W.kalman_cv4(B=B, T=T) for B, T in ((1, 1), (2, 3), (7, 40), (33, 5), (1000, 3), (5000, 2), (20000, 2))],
    *[lambda n=n, m=m, B=B: W.kalman_rand8(B=B, T=4, n=n, m=m, seed=n)
      for n, m, B in ((2, 1, 5), (3, 3, 31), (4, 2, 300), (5, 4, 64), (6, 1, 1), (7, 5, 17), (8, 8, 40), (8, 3, 9000), (12, 7, 9),
                      (16, 6, 20))],
    *[lambda D=D, B=B: W.kalman_highd(B=B, D=D, m=min(D, 8), T=2)
      for D, B in ((9, 5), (16, 3), (20, 5), (24, 1), (24, 300), (32, 5), (32, 700), (40, 2), (48, 3))],
    *[lambda k=k: W.Workload("m", matrix_program(np.random.default_rng(1000 + k)), 0,
                             np.random.default_rng(k).normal(0, 0.5, (3 + 9 * k, 4)), np.zeros(1), np.zeros(4))
      for k in range(30)]])
def test_matrix_records_equal_general(ndvm, oracle_mod, cuda, monkeypatch, make, dtype):
    import torch
    w = make()
    fast, general = _both(ndvm, w, getattr(torch, dtype), monkeypatch)
    for x, y in zip(fast, general):
        np.testing.assert_array_equal(x, y)
    if dtype == "float64":
        idx = np.unique([0, w.B // 2, w.B - 1])
        ol, og, sp = oracle_ref(oracle_mod, w.program, w.params[idx], w.obs)
        ok, rep = rel_check(fast[0][idx], fast[1][idx], ol, og, 1e-12, sp)
        assert ok, rep
    np.testing.assert_array_equal(fast[0], fast[2])


SPARSE = ("(define H (matrix 2 3 1.0 0 0 0 0 2.0)) (define S (matrix 3 3 0 1.0 0 1.0 0 0 0 0 1.0))\n"
          "(model (params a b c) (let* ((X (matrix 3 3 a b 0.5 c a 1.0 b c 2.0)) (Y (matmul S (matmul X S))) (Z (matmul H Y))\n"
          "   (V (matmul Z (matrix 3 1 a 0.0 b))) (Q (matmul (matmul H X) (transpose H))))\n"
          "  (+ (mref V 0 0) (mref V 1 0) (trace Q) (mref Z 1 2) (* c (mref Y 0 1)) (trace (matmul X (zeros 3 3))))))")


def test_constant_zeros_and_non_finite_values(ndvm, cuda, monkeypatch):
    """0 * inf is NaN: a warp that has met an infinity or a NaN takes the constants' zero terms."""
    import torch
    s = np.array([0.0, -0.0, 1.0, -2.5, np.inf, -np.inf, np.nan, 5e-324, 1e308, -1e200])
    a, b, c = np.meshgrid(s, s, s)
    w = W.Workload("sparse", SPARSE, 0, np.stack([a.ravel(), b.ravel(), c.ravel()], 1), np.zeros(1), np.zeros(3))
    fast, general = _both(ndvm, w, torch.float64, monkeypatch)
    for f, g in zip(fast, general):
        np.testing.assert_array_equal(f, g)  # (NaN equals NaN, 0 equals -0)


def test_matrix_records_in_chunks(ndvm, cuda, monkeypatch):
    """A workspace for part of the lanes: the launches over the parts give the same bits."""
    import torch
    w = W.kalman_cv4(B=777, T=9)
    tape = ndvm.trace_build(w.program)
    p, o = torch.tensor(w.params, device="cuda"), torch.tensor(w.obs, device="cuda")
    l1, g1 = ndvm.value_and_grad(tape, p, o)
    per_lane = tape.workspace_bytes(1)
    l2, g2 = ndvm.value_and_grad(tape, p, o, ws_bytes=per_lane * 130)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(l1.cpu().numpy(), l2.cpu().numpy())
    np.testing.assert_array_equal(g1.cpu().numpy(), g2.cpu().numpy())


def _banded(n, band, square=False):
    """A program of banded constants (products with lists, over more than 8 terms from n = 9 on, with a
    block per lane from n = 16 on), scaled by the parameters; its square, whose adjoint is a lane's own."""
    rng = np.random.default_rng(n * 10 + band)
    F = np.where(np.abs(np.subtract.outer(np.arange(n), np.arange(n))) < band, rng.normal(0, 0.4, (n, n)), 0.0)
    lit = " ".join(repr(float(v)) if v else "0" for v in F.ravel())
    eye = " ".join("1.0" if i == j else "0" for i in range(n) for j in range(n))
    ones = " ".join(repr(float(v)) for v in rng.normal(0, 1, n))
    text = (f"(define F (matrix {n} {n} {lit})) (define I (matrix {n} {n} {eye})) (define v (matrix {n} 1 {ones}))\n"
            f"(model (params a b) (let* ((P (m+ (mscale a F) (mscale b I)))"
            f" (Q (matmul F (matmul P (transpose F)))) (R (matmul Q F)) (s (matmul (transpose v) (matmul R v))))"
            f" (let ((z (+ (trace Q) (mref s 0 0)))) {'(* z z)' if square else 'z'})))")
    return text, rng


BANDS = [(8, 3), (9, 1), (9, 2), (12, 3), (15, 4), (16, 5), (24, 2)]


@pytest.mark.parametrize("dtype", ["float64", "float32"])
@pytest.mark.parametrize("n,band", BANDS)
def test_banded_constants_sum_as_dense(ndvm, cuda, monkeypatch, n, band, dtype):
    # products with a banded constant keep the dense sums' chains: a lane's bits do not depend on the
    # number of lanes, which chooses the kernel
    import torch
    text, rng = _banded(n, band)
    w = W.Workload("banded", text, 0, rng.normal(0.5, 0.5, (700, 2)), np.zeros(1), np.zeros(2))
    fast, general = _both(ndvm, w, getattr(torch, dtype), monkeypatch)
    for x, y in zip(fast, general):
        np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("dtype", ["float64", "float32"])
@pytest.mark.parametrize("n,band", BANDS)
def test_banded_constants_and_non_finite_values(ndvm, cuda, monkeypatch, n, band, dtype):
    """Lanes with an infinity, a NaN or an overflow take the zero terms of the lists, of sums over more than
    8 terms, of a block's vote and of a scaling's adjoint; the finite lanes beside them keep their values."""
    import torch
    text, _ = _banded(n, band, square=True)
    v = np.array([0.0, -0.0, 1.0, -2.5, np.inf, -np.inf, np.nan, 1e300, -1e200, 1e38])
    a, b = np.meshgrid(v, v)
    w = W.Workload("banded", text, 0, np.stack([a.ravel(), b.ravel()], 1), np.zeros(1), np.zeros(2))
    fast, general = _both(ndvm, w, getattr(torch, dtype), monkeypatch)
    assert np.isnan(general[1]).any() and np.isfinite(general[1]).any()
    for x, y in zip(fast, general):
        np.testing.assert_array_equal(x, y)  # (NaN equals NaN, 0 equals -0)



@pytest.mark.parametrize("steps", [3, 200])
def test_a_saved_trace(ndvm, oracle_mod, cuda, monkeypatch, steps):
    """The reverse sweep of a long tape reads a trace from the workspace, on both kernels."""
    import torch
    text = ("(model (params a b) (let loop ((i 0) (x a)) (if (= i %d) x (let* ((M (matrix 2 2 x b b a)) (t (trace M)))"
            " (loop (+ i 1) (sin (* t (* 0.5 x))))))))" % steps)
    w = W.Workload("trace", text, 0, np.random.default_rng(steps).normal(0.3, 0.7, (70, 2)), np.zeros(1), np.zeros(2))
    for loss, grad, _ in _both(ndvm, w, torch.float64, monkeypatch):
        ol, og, sp = oracle_ref(oracle_mod, w.program, w.params, w.obs)
        ok, rep = rel_check(loss, grad, ol, og, 1e-12, sp)
        assert ok, rep
