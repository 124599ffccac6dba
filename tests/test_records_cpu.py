"""The compact and matrix records checked without a GPU.

tests/recsim.cpp translates a program's plans to records (compact.cpp), checks every record's
slots, workspace elements, constants and lists, and executes them on the CPU, with 1, 2 and 4
points per pass; tests/plansim.cpp executes the general stream of the same plans.  The two
agree to rounding: the records fuse some reverse rules, and add a data sum's points in another order."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import workloads as W
from conftest import hazard_workloads, matrix_program, oracle_ref, rel_check

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2607_03574_gb300", "csrc")
PLANNER = ["plan.cpp", "tape.cpp", "trace_scheme.cpp", "trace_bytecode.cpp"]


@pytest.fixture(scope="module")
def sims(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    out = tmp_path_factory.mktemp("recsim")
    for name, srcs in (("plansim", PLANNER), ("recsim", PLANNER + ["compact.cpp"])):
        subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, os.path.join(ROOT, "tests", name + ".cpp"),
                        *[os.path.join(CSRC, f) for f in srcs], "-o", str(out / name)], check=True)
    return out


def _run(exe, head, w, B, *args):
    env = {k: v for k, v in os.environ.items() if not k.startswith("NDVM_")}
    body = " ".join(repr(float(x)) for x in w.params[:B].ravel()) + "\n" + " ".join(repr(float(x)) for x in w.obs) + "\n"
    r = subprocess.run([str(exe), *args], input=f"{w.frontend} {B} {w.P} {w.obs.size} {head}\n{body}{w.program}",
                       capture_output=True, text=True, env=env, timeout=300)
    assert r.returncode == 0, (w.name, r.stderr)
    return r.stdout


def _rows(text):
    return np.array([[float.fromhex(t) for t in line.split()] for line in text.strip().splitlines()])


def agree(sims, w, tol=1e-11, B=4):
    """The kinds of the program's two streams ("compact", "matrix" or "none"), after comparing them
    with the general ones: every lane within tol of its largest component, NaN where that is NaN."""
    kinds, B = [], min(B, w.B)
    for value_plan in (0, 1):
        want = _rows(_run(sims / "plansim", "2" if value_plan else "0", w, B))
        for K in (1, 2, 4):
            head, _, rows = _run(sims / "recsim", f"{value_plan} {K}", w, B).partition("\n")
            kind = head.split()[0]
            if K == 1:
                kinds.append(kind)
            if kind == "none":
                break
            got = _rows(rows)
            a, b = (got[:, :1], want[:, :1]) if value_plan else (got, want)
            np.testing.assert_array_equal(np.isnan(a), np.isnan(b), err_msg=w.name)
            with np.errstate(invalid="ignore"):
                scale = np.maximum(np.nanmax(np.abs(np.where(np.isfinite(b), b, 0)), axis=1, keepdims=True), 1e-300)
                err = np.where(np.isfinite(b), np.abs(a - b) / scale, np.where(a == b, 0.0, np.isnan(a) - 1.0))
            assert np.max(np.abs(err), initial=0.0) <= tol, (w.name, value_plan, K, a, b)
    return kinds


def program(text, P, n_obs=0, seed=1, B=4):
    rng = np.random.default_rng(seed)
    return W.Workload("program", text, 0, rng.normal(0.3, 0.7, (B, P)), rng.normal(size=n_obs), np.zeros(P))


def _programs():
    ws = hazard_workloads() + [W.config(1)]
    ws += W.random_exprs(6, B=4, n_points=17, seed=99) + W.control_fuzz(12, B=4, n_points=19, seed=5)
    ws += W.second_client(B=4)
    ws += [W.logistic(B=3), W.kalman_cv4(B=3, T=12), W.kalman_rand8(B=2, T=6), W.kalman_highd(B=2, D=12, m=3, T=3)]
    ws += [W.Workload(f"matrix_{k}", matrix_program(np.random.default_rng(1000 + k)), 0,
                      np.random.default_rng(k).normal(0.0, 0.5, (4, 4)), np.zeros(0), np.zeros(4)) for k in range(40)]
    return ws


PROGRAMS = _programs()


@pytest.mark.parametrize("k", range(len(PROGRAMS)))
def test_records_equal_the_general_stream(sims, k):
    # (a determinant of a nearly singular matrix, and its inverse, magnify the last bits)
    agree(sims, PROGRAMS[k], 1e-7 if PROGRAMS[k].name.startswith("matrix_") else 1e-11)


LONG = "(let loop ((i 0) (x {start})) (if (= i {steps}) x (loop (+ i 1) (+ (* x b) (sin x)))))"


@pytest.mark.parametrize("n,steps,kind", [(0, 3, "compact"), (0, 700, "none"), (1, 700, "none"), (3, 3, "compact")])
def test_a_stream_with_a_loop_is_not_cut_into_chunks(sims, n, steps, kind):
    """A data sum over no points still has its loop's records, and a lane's long stream is read in
    chunks: a stream has the one or the other."""
    w = program(f"(model (params a b) (+ (data-sum {n} 1 (* a (dobs 0))) {LONG.format(start='a', steps=steps)}))", 2, 4)
    assert agree(sims, w) == [kind, kind]
    alone = program(f"(model (params a b) {LONG.format(start='a', steps=steps)})", 2)
    assert agree(sims, alone) == ["compact", "compact"]


ONE_BY_ONE = {  # scalars are 1 x 1 matrices: a record's two operands may both be parameters
    "m+": "(m+ a b)", "m-": "(m- a b)", "mscale": "(mscale a b)", "matmul": "(matmul a b)", "one": "(matmul a a)",
    "fold": "(m+ b (matmul a b))", "const": "(m- (mscale 3.0 b) (m+ a 2.0))", "inv": "(matmul (inv a) b)",
    "det": "(mscale (det a) (logdet (mscale 2.0 (matmul b b))))",
}


@pytest.mark.parametrize("name", sorted(ONE_BY_ONE))
def test_parameters_as_matrix_operands(sims, name):
    w = program(f"(model (params a b) (let* ((Z {ONE_BY_ONE[name]})) (+ (* Z Z) (trace (mscale Z b)))))", 2)
    assert agree(sims, w) == ["matrix", "matrix"]


@pytest.mark.parametrize("big,lists", [("1e999", False), ("-1e999", False), ("1e39", False), ("1e38", True)])
@pytest.mark.parametrize("order", ["(matmul S D)", "(matmul D S)"])
def test_zeros_of_a_constant_times_an_infinite_constant(sims, order, big, lists):
    """0 * inf is NaN: a product of two constants leaves out no term when one holds an infinity.  1e39 is
    one in binary32, whose records have the same lists of the terms to take."""
    w = program(f"(define S (matrix 2 2 1.5 0.0 0.0 2.0)) (define D (matrix 2 2 {big} 2.0 3.0 4.0))"
                f"(model (params a b) (trace (mscale a {order})))", 2)
    assert agree(sims, w) == ["matrix", "matrix"]
    head = _run(sims / "recsim", "0 1", w, 1).split("\n")[0]
    assert (int(head.split()[1]) > 0) == lists


TRACES = ("(model (params a b) (let loop ((i 0) (x a)) (if (= i {steps}) x "
          "(let* ((M (matrix 2 2 x b b a)) (t (trace M))) (loop (+ i 1) (sin (* t (* 0.5 x))))))))")


@pytest.mark.parametrize("steps", [3, 200])
def test_a_trace_that_the_reverse_sweep_reads_is_saved(sims, oracle_mod, steps):
    """A long tape's forward values reach the reverse sweep through the workspace, a trace's too."""
    w = program(TRACES.format(steps=steps), 2)
    assert agree(sims, w) == ["matrix", "matrix"]
    got = _rows(_run(sims / "plansim", "0", w, w.B))
    loss, grad, spread = oracle_ref(oracle_mod, w.program, w.params, w.obs)
    ok, rep = rel_check(got[:, 0], got[:, 1:], loss, grad, 1e-12, spread)
    assert ok, rep


def test_a_seed_apart_from_its_loop_is_refused(sims):
    """Points past the last one are told by the body's seed, set just ahead of the loop: a stream in which
    it is not recognised as the loop's has no compact form."""
    w = program("(model (params a b) (data-sum 3 2 (let ((r (- (* a (exp (* b (dobs 0)))) (dobs 1)))) (* r r))))", 2, 6)
    assert agree(sims, w) == ["compact", "compact"]
    kinds = [_run(sims / "recsim", f"{stream} 1", w, 1, "apart").split()[0] for stream in (0, 1)]
    assert kinds == ["none", "compact"]  # (the value plan's loop has no seed)
