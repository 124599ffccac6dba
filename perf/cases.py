"""The calls whose speed is measured: what users of the tape replay have it do, through the
package's public entry points.

A case is one program (or a population of programs), a number of parameter lanes, a data
type and the entry point that runs it:

  model     decay     a exp(-b t) + c fitted to points (a data sum; the smallest programs)
            exprs     random expression programs of + - * / exp log sin pow (program search)
            logistic  stack bytecode, explicit Euler steps (long scalar chains)
            cv4       4-state constant-velocity Kalman likelihood
            kalman    n-state Kalman likelihood, random stable transition, m observations
  call      grad      value_and_grad on device tensors
            forward   forward (no gradient: scoring a population)
            multi     value_and_grad_multi (one call for a population of programs)
            streams   value_and_grad per program, the programs spread over streams
            host      value_and_grad_host (numpy in, numpy out)
            op        loss_op inside torch autograd (a calibration step's forward and backward)

A case's program is made from its `text_seed`; parameters and observations come from the
seed that `prepare` is given.
"""
import math

import numpy as np
import torch

import paper_2607_03574_gb300 as nd

STREAMS = 8


# ------------------------------------------------------------------------------ the cases
def listed():
    return [
        # a user's first fit: few lanes, few points, one call after another (latency, launches)
        _c("decay_64", "decay", "grad", 64, "f64", points=50),
        # the same kind of fit over a wide, ragged population in single precision
        _c("decay_f32_wide", "decay", "grad", 50001, "f32", points=333),
        # program search, early rounds: many candidate programs, few lanes each, one call
        _c("search_batched", "exprs", "multi", 64, "f64", points=256, programs=24, text_seed=11),
        # program search at the repository's headline shape: 4096 lanes, 256 points per program
        _c("search_streams", "exprs", "streams", 4096, "f64", points=256, programs=24, text_seed=12),
        # one candidate scored from host data, odd sizes (numpy in, numpy out)
        _c("expr_host", "exprs", "host", 1500, "f64", points=201, programs=1, text_seed=13),
        # ODE fit: 1000 Euler steps in stack bytecode, the repository's full size
        _c("logistic_f64", "logistic", "grad", 16384, "f64", steps=1000, every=10),
        _c("logistic_f32", "logistic", "grad", 16384, "f32", steps=1000, every=10),
        # tracking filter likelihood, the repository's full size, and its scoring pass
        _c("cv4_f64", "cv4", "grad", 8192, "f64", steps=200),
        _c("cv4_forward", "cv4", "forward", 3001, "f64", steps=200),
        # calibration step through torch autograd: a small population, 80 steps
        _c("cv4_op_step", "cv4", "op", 256, "f64", steps=80),
        # the largest: 8-state filters
        _c("kalman8", "kalman", "grad", 16384, "f64", steps=120, n=8, m=3, text_seed=14),
        # high-dimensional population (a lane fills an SM's shared memory)
        _c("kalman64", "kalman", "grad", 152, "f64", steps=10, n=64, m=8, text_seed=15),
    ]


def _c(name, model, call, lanes, dtype, points=0, programs=1, steps=0, every=0, n=0, m=0, text_seed=0):
    case = {"name": name, "model": model, "call": call, "lanes": lanes, "dtype": dtype, "points": points,
            "programs": programs, "steps": steps, "every": every, "n": n, "m": m, "text_seed": text_seed}
    return case


def draw(rng):
    """One more case of the listed ones' ranges: every model, entry point and data type, lanes
    from 1 up, odd sizes; no more work than the largest listed case."""
    most = max(work(c)["flops"] for c in listed())
    while True:
        model = rng.choice(["decay", "exprs", "exprs", "logistic", "cv4", "kalman"])
        call = rng.choice(["grad", "grad", "grad", "forward", "host", "op"])
        programs = points = steps = every = n = m = 0
        lanes = _log(rng, 1, 60000)
        programs = 1
        if model == "decay":
            points = _log(rng, 5, 1000)
        elif model == "exprs":
            call = rng.choice([call, "multi", "streams"])
            points = _log(rng, 16, 1024)
            if call in ("multi", "streams"):
                programs = rng.randint(2, 24)
                lanes = _log(rng, 1, 5000)
        elif model == "logistic":
            every = rng.randint(1, 12)
            steps = every * _log(rng, 2, max(2, 1000 // every))
            lanes = _log(rng, 1, 20000)
        else:
            steps = _log(rng, 3, 200)
            lanes = _log(rng, 1, 16384)
            if model == "kalman":
                n = rng.choice([2, 3, 5, 6, 7, 8, 8, 12, 16, 24, 32, 48, 64])
                m = rng.randint(1, min(n, 8))
                if n > 16:
                    steps = _log(rng, 2, 10)
                    lanes = _log(rng, 1, 400)
        case = _c("", model, call, lanes, rng.choice(["f64", "f64", "f32"]), points, programs, steps, every, n, m,
                  rng.randrange(1 << 20))
        del case["name"]
        if work(case)["flops"] <= most:
            return case


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


# --------------------------------------------------------------------------- program texts
def _num(x):
    s = repr(float(x))
    return s if ("." in s or "e" in s) else s + ".0"


def _decay_text(points):
    return (f"(model (params a b c) (/ (data-sum {points} 2\n"
            "  (let ((r (- (+ (* a (exp (- (* b (dobs 0))))) c) (dobs 1)))) (* r r)))\n"
            f" {_num(points)}))\n")


def _logistic_text(n_obs, every):
    return "\n".join([
        "PARAM 0", "STORE 0", "PARAM 1", "STORE 1", "PUSH 0.1", "STORE 2", "PUSH 0.0", "STORE 3",
        f"LOOP {n_obs}", f"  LOOP {every}",
        "    LOAD 2", "    LOAD 0", "    LOAD 2", "    MUL", "    PUSH 1.0", "    LOAD 2", "    LOAD 1", "    DIV",
        "    SUB", "    MUL", "    PUSH 0.01", "    MUL", "    ADD", "    STORE 2", "  END",
        "  LOAD 3", "  LOAD 2", "  OBSN", "  SUB", "  DUP", "  MUL", "  ADD", "  STORE 3", "END",
        "LOAD 3", f"PUSH {_num(n_obs)}", "DIV"]) + "\n"


_FILTER = """(define (kalman-nll Q R P0 T)
  (let loop ((t 0) (x (zeros {n} 1)) (P P0) (nll 0.0))
    (if (= t T)
        nll
        (let* ((xp (matmul F x))
               (Pp (m+ (matmul (matmul F P) (transpose F)) Q))
               (v (m- (obs-vec (* {m} t) {m}) (matmul H xp)))
               (PHt (matmul Pp (transpose H)))
               (S (m+ (matmul H PHt) R))
               (Si (inv S))
               (K (matmul PHt Si))
               (xn (m+ xp (matmul K v)))
               (Pn (m- Pp (matmul K (matmul H Pp))))
               (term (* 0.5 (+ (logdet S) (mref (matmul (transpose v) (matmul Si v)) 0 0) {c}))))
          (loop (+ t 1) xn Pn (+ nll term))))))
"""


def _matrix(M):
    return f"(matrix {M.shape[0]} {M.shape[1]} {' '.join(_num(v) for v in M.reshape(-1))})"


def _filter_text(F, H, steps):
    n, m = F.shape[0], H.shape[0]
    return (f"(define F {_matrix(F)})\n(define H {_matrix(H)})\n"
            + _FILTER.format(n=n, m=m, c=_num(m * math.log(2 * math.pi))))


_CV4_F = np.array([[1, 0, 1, 0], [0, 1, 0, 1], [0, 0, 1, 0], [0, 0, 0, 1]], dtype=float)
_CV4_H = np.array([[1, 0, 0, 0], [0, 1, 0, 0]], dtype=float)


def _cv4_text(steps):
    return _filter_text(_CV4_F, _CV4_H, steps) + (
        "(model (params lqx lqy lrx lry)\n"
        "  (let* ((qx (exp (* 2.0 lqx))) (qy (exp (* 2.0 lqy))) (rx (exp (* 2.0 lrx))) (ry (exp (* 2.0 lry)))\n"
        "         (Q (matrix 4 4 (/ qx 3.0) 0 (/ qx 2.0) 0  0 (/ qy 3.0) 0 (/ qy 2.0)\n"
        "                        (/ qx 2.0) 0 qx 0  0 (/ qy 2.0) 0 qy))\n"
        "         (R (matrix 2 2 rx 0 0 ry)))\n"
        f"    (kalman-nll Q R (mscale 10.0 (identity 4)) {steps})))\n")


def _kalman_system(case):
    rng = np.random.default_rng(case["text_seed"])
    n, m = case["n"], case["m"]
    A = rng.normal(0.0, 1.0, (n, n))
    F = A * (0.95 / float(np.max(np.abs(np.linalg.eigvals(A)))))
    H = np.zeros((m, n))
    H[:, :m] = np.eye(m)
    return F, H


def _diag_text(size, names):
    rows = []
    for i, name in enumerate(names):
        row = ["0"] * size
        row[i] = f"(exp (* 2.0 {name}))"
        rows.append(" ".join(row))
    return f"(matrix {size} {size} " + "\n ".join(rows) + ")"


def _kalman_text(case):
    F, H = _kalman_system(case)
    n, m, T = case["n"], case["m"], case["steps"]
    head = _filter_text(F, H, T)
    if n > 16:  # one parameter per noise covariance
        return head + ("(model (params lq lr lp0) (kalman-nll "
                       f"(mscale (exp (* 2.0 lq)) (identity {n})) (mscale (exp (* 2.0 lr)) (identity {m}))\n"
                       f" (mscale (exp (* 2.0 lp0)) (identity {n})) {T}))\n")
    q, r = [f"lq{i}" for i in range(n)], [f"lr{i}" for i in range(m)]
    return head + (f"(model (params {' '.join(q + r)} lp0) (kalman-nll {_diag_text(n, q)}\n {_diag_text(m, r)}\n"
                   f" (mscale (exp (* 2.0 lp0)) (identity {n})) {T}))\n")


def _noise_params(case):
    """Centre of the lanes' parameters (logarithms of standard deviations)."""
    if case["model"] == "cv4":
        return np.log(np.array([0.5, 0.4, 1.0, 0.8]))
    n, m = case["n"], case["m"]
    if n > 16:
        return np.array([math.log(0.2), math.log(0.5), 0.0])
    q = np.random.default_rng(case["text_seed"] + 1).uniform(0.1, 0.3, n)
    return np.concatenate([np.log(q), np.full(m, math.log(0.5)), [0.0]])


# Random expressions.  Divisors become 1 + d^2, exponents a / (1 + a^2), logarithms log|1 + a^2|,
# and a program is kept only if every intermediate stays below 1e4 in size around its constants.
def _tree(rng, depth, state):
    def leaf():
        if (rng.random() < 0.5 or state[0] == 0) and state[0] < 8 and rng.random() < 0.6:
            state[0] += 1
            return ("c", state[0] - 1)
        if state[0] > 0 and rng.random() < 0.3:
            return ("c", int(rng.integers(0, state[0])))
        return ("x",)

    if depth >= 6 or (depth > 0 and rng.random() < 0.15 + 0.85 * (depth / 6) ** 2):
        return leaf()
    if rng.random() < 0.65:
        op = "+-*/"[int(rng.integers(0, 4))]
        return (op, _tree(rng, depth + 1, state), _tree(rng, depth + 1, state))
    op = ("exp", "log", "sin", "pow")[int(rng.integers(0, 4))]
    if op == "pow":
        return (op, _tree(rng, depth + 1, state), int(rng.integers(2, 4)))
    return (op, _tree(rng, depth + 1, state))


def _subtrees(e):
    return [s for s in e[1:] if isinstance(s, tuple)]


def _count(e):
    return 1 + sum(_count(s) for s in _subtrees(e))


def _has_x(e):
    return e[0] == "x" or any(_has_x(s) for s in _subtrees(e))


def _evaluate(e, x, th, seen, lib):
    """The tree on points x ([1, N]) and constants th ([B, P]), in numpy or torch."""
    def sub(k):
        return _evaluate(e[k], x, th, seen, lib)

    k = e[0]
    if k == "x":
        v = x + 0 * th[:, :1]
    elif k == "c":
        v = th[:, e[1]:e[1] + 1] + 0 * x
    elif k in "+-*":
        a, b = sub(1), sub(2)
        v = a + b if k == "+" else a - b if k == "-" else a * b
    elif k == "/":
        a, b = sub(1), sub(2)
        v = a / (1.0 + b * b)
    elif k == "exp":
        a = sub(1)
        v = lib.exp(a / (1.0 + a * a))
    elif k == "log":
        a = sub(1)
        v = lib.log(abs(1.0 + a * a))
    elif k == "sin":
        v = lib.sin(sub(1))
    else:
        v = sub(1) ** e[2]
    if seen is not None:
        seen.append(float(np.max(np.abs(v))))
    return v


def _expr_text(e, fresh):
    def name():
        fresh[0] += 1
        return f"g{fresh[0]}"

    k = e[0]
    if k == "x":
        return "x"
    if k == "c":
        return f"t{e[1]}"
    if k in "+-*":
        return f"({k} {_expr_text(e[1], fresh)} {_expr_text(e[2], fresh)})"
    if k == "/":
        a, b, v = _expr_text(e[1], fresh), _expr_text(e[2], fresh), name()
        return f"(let (({v} {b})) (/ {a} (+ 1.0 (* {v} {v}))))"
    a = _expr_text(e[1], fresh)
    if k == "sin":
        return f"(sin {a})"
    if k == "pow":
        return f"(pow {a} {e[2]})"
    v = name()
    if k == "exp":
        return f"(let (({v} {a})) (exp (/ {v} (+ 1.0 (* {v} {v})))))"
    return f"(let (({v} {a})) (log (abs (+ 1.0 (* {v} {v})))))"


def _expr_programs(case):
    """[(tree, centre of the constants)] of the case's programs."""
    rng = np.random.default_rng(case["text_seed"])
    out = []
    while len(out) < case["programs"]:
        state = [0]
        tree = _tree(rng, 0, state)
        if state[0] < 1 or not _has_x(tree) or _count(tree) < 4:
            continue
        theta = rng.uniform(-2.0, 2.0, state[0])
        seen = []
        with np.errstate(all="ignore"):
            _evaluate(tree, np.linspace(-2.0, 2.0, 65)[None], theta + rng.normal(0.0, 0.5, (48, state[0])), seen, np)
        if np.all(np.isfinite(seen)) and max(seen) < 1e4:
            out.append((tree, theta))
    return out


def _expr_program_text(tree, P, points):
    return (f"(model (params {' '.join(f't{k}' for k in range(P))}) (/ (data-sum {points} 2\n"
            f" (let* ((x (dobs 0)) (r (- {_expr_text(tree, [0])} (dobs 1)))) (* r r))) {_num(points)}))\n")


# ---------------------------------------------------------------------------------- inputs
def _simulate(rng, F, H, q_std, r_std, p_std, T):
    n, m = H.shape[1], H.shape[0]
    x, ys = p_std * rng.normal(size=n), []
    for _ in range(T):
        x = F @ x + q_std * rng.normal(size=n)
        ys.append(H @ x + r_std * rng.normal(size=m))
    return np.concatenate(ys)


def _inputs(case, seed):
    """[(program text, front end, params [B, P], obs [n])] in float64 numpy, one per program."""
    rng = np.random.default_rng([seed, 77])
    B, model = case["lanes"], case["model"]
    if model == "decay":
        N = case["points"]
        t = rng.uniform(0.0, 5.0, N)
        obs = np.stack([t, 1.3 * np.exp(-0.8 * t) + 0.9 + rng.normal(0.0, 0.05, N)], 1).reshape(-1)
        return [(_decay_text(N), nd.FE_SCHEME, rng.normal(1.0, 0.3, (B, 3)), obs)]
    if model == "exprs":
        out, N = [], case["points"]
        for tree, theta in _expr_programs(case):
            x = rng.uniform(-2.0, 2.0, N)
            y = _evaluate(tree, x[None], theta[None], None, np)[0] + rng.normal(0.0, 0.05, N)
            out.append((_expr_program_text(tree, theta.size, N), nd.FE_SCHEME,
                        theta + rng.normal(0.0, 0.3, (B, theta.size)), np.stack([x, y], 1).reshape(-1)))
        return out
    if model == "logistic":
        n_obs, x, ys = case["steps"] // case["every"], 0.1, []
        for _ in range(n_obs):
            for _ in range(case["every"]):
                x = x + 0.01 * (0.8 * x * (1.0 - x))
            ys.append(x)
        obs = np.array(ys) + rng.normal(0.0, 0.01, n_obs)
        params = np.array([0.8, 1.0]) * np.exp(0.25 * rng.normal(size=(B, 2)))
        return [(_logistic_text(n_obs, case["every"]), nd.FE_BYTECODE, params, obs)]
    centre = _noise_params(case)
    if model == "cv4":
        text, (F, H) = _cv4_text(case["steps"]), (_CV4_F, _CV4_H)
        std = np.exp(centre)
        obs = _simulate(rng, F, H, np.array([0.58, 0.58, 1, 1]) * std[[0, 1, 0, 1]], std[2:], 3.0, case["steps"])
        spread = 0.5
    else:
        text, (F, H) = _kalman_text(case), _kalman_system(case)
        n, m, std = case["n"], case["m"], np.exp(centre)
        q, r = (std[0], std[1]) if n > 16 else (std[:n], std[n:n + m])
        obs = _simulate(rng, F, H, q, r, 1.0, case["steps"])
        spread = 0.3 if n > 16 else 0.5
    return [(text, nd.FE_SCHEME, centre + rng.normal(0.0, spread, (B, centre.size)), obs)]


def prepare(case, seed):
    np_type = np.float32 if case["dtype"] == "f32" else np.float64
    state = {"call": case["call"], "tapes": [], "params": [], "obs": []}
    for text, frontend, params, obs in _inputs(case, seed):
        state["tapes"].append(nd.trace_build(text, frontend))
        params, obs = params.astype(np_type), obs.astype(np_type)
        if case["call"] != "host":
            params, obs = torch.from_numpy(params).cuda(), torch.from_numpy(obs).cuda()
        if case["call"] == "op":
            params.requires_grad_(True)
        state["params"].append(params)
        state["obs"].append(obs)
    if case["call"] == "streams":
        state["streams"] = _shared_streams()
    if case["call"] == "op":
        state["op"] = nd.loss_op(state["tapes"][0])
    return state


_STREAMS = []


def _shared_streams():
    """A program's worker streams, made once."""
    while len(_STREAMS) < STREAMS:
        _STREAMS.append(torch.cuda.Stream())
    return _STREAMS


def run(state):
    call, tapes, params, obs = state["call"], state["tapes"], state["params"], state["obs"]
    if call == "grad":
        return [nd.value_and_grad(t, p, o) for t, p, o in zip(tapes, params, obs)]
    if call == "forward":
        return [nd.forward(t, p, o) for t, p, o in zip(tapes, params, obs)]
    if call == "multi":
        return nd.value_and_grad_multi(tapes, params, obs)
    if call == "host":
        return [nd.value_and_grad_host(t, p, o) for t, p, o in zip(tapes, params, obs)]
    if call == "op":
        loss = state["op"](params[0], obs[0])
        (grad,) = torch.autograd.grad(loss.sum(), params[0])
        return loss.detach(), grad
    # streams: each program on its stream, the caller's stream before and after them all
    here, out = torch.cuda.current_stream(), []
    for s in state["streams"]:
        s.wait_stream(here)
    for k, (t, p, o) in enumerate(zip(tapes, params, obs)):
        out.append(nd.value_and_grad(t, p, o, stream=state["streams"][k % STREAMS]))
    for s in state["streams"]:
        here.wait_stream(s)
    return out


# -------------------------------------------------------------------- what a pass must do
def _tree_flops(e):
    """Operations of an expression's forward sweep per point, and of its reverse sweep."""
    k = e[0]
    f, r = {"x": (0, 0), "c": (0, 1), "+": (1, 1), "-": (1, 1), "*": (1, 4), "/": (3, 8), "exp": (14, 7),
            "log": (15, 8), "sin": (12, 3), "pow": (2, 4)}[k]
    for s in _subtrees(e):
        a, b = _tree_flops(s)
        f, r = f + a, r + b
    return f, r


def work(case):
    """Bytes: parameters, observations and outputs once.  Operations: one per addition and
    multiplication (a fused one counts two), about ten per exp, log or sin, of the forward
    sweep and, unless the call is `forward`, of the reverse sweep."""
    B, size = case["lanes"], 4 if case["dtype"] == "f32" else 8
    grad = case["call"] != "forward"
    flops = bytes_ = 0.0
    if case["model"] == "decay":
        progs = [(3, 2 * case["points"], case["points"] * (18 if not grad else 30))]
    elif case["model"] == "exprs":
        progs = []
        for tree, theta in _expr_programs(case):
            f, r = _tree_flops(tree)
            progs.append((theta.size, 2 * case["points"], case["points"] * (f + 3 + (r + 1 if grad else 0))))
    elif case["model"] == "logistic":
        progs = [(2, case["steps"] // case["every"], case["steps"] * (6 + (12 if grad else 0)))]
    else:
        n, m = (4, 2) if case["model"] == "cv4" else (case["n"], case["m"])
        P = _noise_params(case).size
        products = 2 * (2 * n ** 3 + n * n + 2 * n * n * m + n * m * (m + n) + n * m * m + 2 * n * m + m * m)
        fwd = products + 2 * n * n + m * m + 3 * m ** 3
        progs = [(P, m * case["steps"], case["steps"] * fwd * (3 if grad else 1))]
    for P, n_obs, per_lane in progs:
        flops += float(B) * per_lane
        bytes_ += size * (n_obs + B * (P + 1 + (P if grad else 0)))
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    # errors against `exact` reach 1e-6 and 3e-15; a few lanes whose gradient cancels show more
    return {"rel": 4e-5} if case["dtype"] == "f32" else {"rel": 2e-13}


# --------------------------------------------------------------------------- 64-bit answers
def _exact_loss(case, tree, th, obs):
    model = case["model"]
    if model in ("decay", "exprs"):
        x, y = obs[0::2][None], obs[1::2][None]
        f = (th[:, :1] * torch.exp(-(th[:, 1:2] * x)) + th[:, 2:3]) if model == "decay" else \
            _evaluate(tree, x, th, None, torch)
        return ((f - y) ** 2).sum(1) / case["points"]
    if model == "logistic":
        r, K = th[:, 0], th[:, 1]
        x, acc = torch.full_like(r, 0.1), torch.zeros_like(r)
        for k in range(obs.numel()):
            for _ in range(case["every"]):
                x = x + 0.01 * (r * x * (1.0 - x / K))
            acc = acc + (x - obs[k]) ** 2
        return acc / obs.numel()
    like = {"dtype": th.dtype, "device": th.device}
    var = torch.exp(2.0 * th)
    if model == "cv4":
        F, H = torch.tensor(_CV4_F, **like), torch.tensor(_CV4_H, **like)
        shape = torch.tensor([[1 / 3, 0.5], [0.5, 1.0]], **like)
        ex = torch.tensor([[1.0, 0.0], [0.0, 0.0]], **like)
        ey = torch.tensor([[0.0, 0.0], [0.0, 1.0]], **like)
        Q = var[:, 0, None, None] * torch.kron(shape, ex) + var[:, 1, None, None] * torch.kron(shape, ey)
        R, P0 = torch.diag_embed(var[:, 2:]), 10.0 * torch.eye(4, **like).expand(th.shape[0], 4, 4)
    else:
        n, m = case["n"], case["m"]
        F, H = (torch.tensor(M, **like) for M in _kalman_system(case))
        eye_n, eye_m = torch.eye(n, **like), torch.eye(m, **like)
        if n > 16:
            Q, R, P0 = (var[:, k, None, None] * e for k, e in ((0, eye_n), (1, eye_m), (2, eye_n)))
        else:
            Q, R = torch.diag_embed(var[:, :n]), torch.diag_embed(var[:, n:n + m])
            P0 = var[:, -1, None, None] * eye_n
    n, m = F.shape[0], H.shape[0]
    x, P = torch.zeros(th.shape[0], n, 1, **like), P0
    nll = torch.zeros(th.shape[0], **like)
    for t in range(case["steps"]):
        xp, Pp = F @ x, F @ P @ F.T + Q
        v = obs[m * t:m * (t + 1), None] - H @ xp
        PHt = Pp @ H.T
        S = H @ PHt + R
        Si = torch.linalg.inv(S)
        K = PHt @ Si
        x, P = xp + K @ v, Pp - K @ (H @ Pp)
        quad = (v.transpose(1, 2) @ (Si @ v))[:, 0, 0]
        nll = nll + 0.5 * (torch.log(torch.linalg.det(S)) + quad + m * math.log(2 * math.pi))
    return nll


def exact(case, seed):
    np_type = np.float32 if case["dtype"] == "f32" else np.float64
    trees = [t for t, _ in _expr_programs(case)] if case["model"] == "exprs" else [None]
    grad, losses, grads = case["call"] != "forward", [], []
    device = "cuda" if torch.cuda.is_available() else "cpu"
    for (_, _, params, obs), tree in zip(_inputs(case, seed), trees):
        th = torch.from_numpy(params.astype(np_type).astype(np.float64)).to(device)
        o = torch.from_numpy(obs.astype(np_type).astype(np.float64)).to(device)
        parts_l, parts_g = [], []
        for part in th.split(4096 if case["model"] != "logistic" else 32768):  # bounded memory
            part = part.clone().requires_grad_(grad)
            with torch.set_grad_enabled(grad):
                loss = _exact_loss(case, tree, part, o)
            if grad:
                parts_g.append(torch.autograd.grad(loss.sum(), part)[0])
            parts_l.append(loss.detach())
        losses.append(torch.cat(parts_l))
        if grad:
            grads.append(torch.cat(parts_g))
    if case["call"] == "forward":
        return losses
    if case["call"] == "multi":
        return losses, grads
    if case["call"] == "op":
        return losses[0], grads[0]
    return list(zip(losses, grads))
