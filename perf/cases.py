"""Workloads that a user of the solver runs, one pass each.

A pass goes through the package's public entry points (`Solver`, `batch_solve`)
the way a user's program does.  The sizes are those of this repository's own
configurations and tests: the 1-D Poisson problem (16 subdomains, K = 64, 2000
points), the damped oscillator (levels 1..64, K = 96, 20000 points), the 2-D
multilevel Poisson problem (levels 1..16, K = 128, 400^2 points), the large 2-D
problem (levels 1..64, K = 64, 2048^2 points) and uneven single-level 2-D
instances.  `draw` varies them over the ranges that these stand for.

Solves run a fixed number of LSQR iterations from a cold start: an LSQR iterate
of a few steps is a well-determined function of the inputs, where a converged
one is not (rounding steers which Krylov direction enters next).  For the same
reason the block-Jacobi shift is 1e-2: FP32 panels then determine the iterates
to FP32 accuracy, where the factors of a far smaller shift amplify the panels'
own rounding a thousandfold; the work does not depend on it.  Results computed
from FP32 panels are kept as FP32, those from FP64 or FP32-pair panels as FP64.
"""
import math
import types

import numpy as np
import torch

import paper_2409_01949_gb300 as E

DEV = "cuda"
#: LSQR steps of a whole fit, of a block-Jacobi solve and of a batched instance
FIT_ITERS, SOLVE_ITERS, BATCH_ITERS = 4, 20, 20
#: block-Jacobi shift of FP32 panels, and the rank cut of the direct solver
SHIFT, QR_RCOND = 1e-2, 1e-13
PREC = {"fp64": E.FP64, "fp32": E.FP32, "mixed": E.MIXED, "df32": E.DF32}


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # evaluating a fitted 1-D model at a plot's worth of points: the
        # smallest call, launch and host latency
        dict(name="eval_1d", kind="eval", dim=1, levels="16", K=64, points=1000),
        # a fine output grid of the large 2-D model (512^2 points)
        dict(name="eval_2d_large", kind="eval", dim=2, levels="1,2,4,8,16,32,64", K=64,
             points=262144),
        # a whole call on the smallest problem, FP64 throughout, in the paper's
        # protocol (unpreconditioned LSQR): create, assemble, solve, evaluate
        dict(name="fit_poisson_1d", kind="fit", pde="poisson", dim=1, levels="16", K=64, n=2000,
             precision="fp64", iters=FIT_ITERS, points=1000),
        # the direct solver on the same system: dense column-pivoted QR
        dict(name="qr_poisson_1d", kind="qr", pde="poisson", dim=1, levels="16", K=64, n=2000,
             precision="fp64", rcond=QR_RCOND, points=1000),
        # a new time interval or operator: the multilevel oscillator assembled
        # to FP32-pair panels and the first LSQR steps on it
        dict(name="fit_oscillator", kind="fit", pde="oscillator", dim=1,
             levels="1,2,4,8,16,32,64", K=96, n=20000, precision="df32", iters=FIT_ITERS,
             points=1000),
        # one system assembled anew (new points or operator), FP32 panels
        dict(name="assemble_2d_multilevel", kind="assemble", pde="poisson", dim=2,
             levels="1,2,4,8,16", K=128, n=400, precision="fp32"),
        # the same with FP64 panels
        dict(name="assemble_2d_fp64", kind="assemble", pde="poisson", dim=2,
             levels="1,2,4,8,16", K=128, n=400, precision="fp64"),
        # block-Jacobi LSQR on an assembled 2-D system, then the model on the
        # 96^2 test grid
        dict(name="solve_2d_multilevel", kind="solve", pde="poisson", dim=2, levels="1,2,4,8,16",
             K=128, n=400, precision="fp32", iters=SOLVE_ITERS, shift=SHIFT),
        # the same on the largest configuration (4.2M rows, 350k columns)
        dict(name="solve_2d_large", kind="solve", pde="poisson", dim=2,
             levels="1,2,4,8,16,32,64", K=64, n=2048, precision="fp32", iters=SOLVE_ITERS,
             shift=SHIFT),
        # the normal-equations blocks on the tensor cores (BF16 operands): every
        # block, then the diagonal ones and one row of neighbours read back
        dict(name="gram_2d_multilevel", kind="gram", pde="poisson", dim=2, levels="1,2,4,8,16",
             K=128, n=400, precision="mixed"),
        # many small problems of uneven size in one call, from host arrays
        dict(name="batch_2d", kind="batch", instances=24, n_sub=16, K=128, n=256, iters=BATCH_ITERS,
             shift=SHIFT),
        # one training step's gradient of the learned preconditioner's network
        dict(name="network_gradient", kind="network", pde="poisson", dim=2, levels="1,2,4,8,16",
             K=64, n=128, precision="fp32", batch=8),
    ]


#: the ranges that the listed cases stand for
LEVELS_1D = ("8", "16", "20", "32", "1,2,4,8,16", "1,2,4,8,16,32", "1,2,4,8,16,32,64")
LEVELS_2D = ("4", "8", "13", "16", "1,2,4", "1,2,4,8", "1,2,4,8,16", "1,2,4,8,16,32")
FEATURES = (24, 32, 40, 48, 64, 80, 96, 128)


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed cases' kinds and ranges."""
    kind = rng.choice(("eval", "eval", "fit", "fit", "qr", "assemble", "solve", "solve", "gram",
                       "gram", "batch", "network"))
    if kind == "eval":
        dim = rng.choice((1, 2))
        c = dict(kind=kind, dim=dim, levels=rng.choice(LEVELS_1D if dim == 1 else LEVELS_2D),
                 K=rng.choice(FEATURES + (12, 33, 100)), points=_logint(rng, 300, 200000),
                 delta=rng.choice((2.0, 2.0, 2.5, 2.9)))
    elif kind == "fit":
        pde = rng.choice(("poisson", "oscillator"))
        c = dict(kind=kind, pde=pde, dim=1, levels=rng.choice(LEVELS_1D), K=rng.choice(FEATURES),
                 n=_logint(rng, 500, 20000), precision=rng.choice(("fp64", "df32")),
                 iters=FIT_ITERS, points=_logint(rng, 300, 3000))
    elif kind == "qr":
        J, K = rng.choice(((8, 24), (8, 64), (16, 33), (16, 64), (20, 12), (20, 32)))
        c = dict(kind=kind, pde="poisson", dim=1, levels=str(J), K=K, n=_logint(rng, 1100, 2000),
                 precision="fp64", rcond=QR_RCOND, points=_logint(rng, 300, 3000))
    elif kind == "assemble":
        c = dict(kind=kind, pde="poisson", dim=2, levels=rng.choice(LEVELS_2D),
                 K=rng.choice(FEATURES), n=_logint(rng, 64, 400),
                 precision=rng.choice(("fp32", "fp32", "fp64")),
                 delta=rng.choice((2.0, 2.0, 2.9)))
    elif kind == "solve":
        K = rng.choice((32, 48, 64, 96, 128))
        n = _logint(rng, 100, 900)
        # the finest level keeps several points per feature in a support
        fits = [v for v in LEVELS_2D if (2.0 * n / int(v.split(",")[-1])) ** 2 >= 4 * K]
        c = dict(kind=kind, pde="poisson", dim=2, levels=rng.choice(fits), K=K, n=n,
                 precision="fp32", iters=SOLVE_ITERS, shift=SHIFT)
    elif kind == "gram":
        c = dict(kind=kind, pde="poisson", dim=2, levels=rng.choice(LEVELS_2D),
                 K=rng.choice((32, 48, 64, 80, 96, 128)), n=_logint(rng, 64, 400),
                 precision="mixed")
    elif kind == "batch":
        c = dict(kind=kind, instances=rng.randint(4, 20), n_sub=rng.choice((6, 9, 12)),
                 K=rng.choice((32, 64, 128)), n=_logint(rng, 128, 256), iters=BATCH_ITERS,
                 shift=SHIFT)
    else:
        c = dict(kind=kind, pde="poisson", dim=2, levels=rng.choice(LEVELS_2D[:-1]),
                 K=rng.choice((32, 48, 64, 96, 128)), n=_logint(rng, 64, 160), precision="fp32",
                 batch=rng.randint(1, 8))
    return c


def _levels(case):
    return [int(v) for v in case["levels"].split(",")]


def _delta(case):
    return case.get("delta", 2.0)


def _subdomains(case):
    return sum(v ** case["dim"] for v in _levels(case))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _generator(seed, device=DEV):
    return torch.Generator(device=device).manual_seed(int(seed) & 0x7FFFFFFF)


def _model_seed(seed):
    return (int(seed) * 2654435761 + 12345) & 0x7FFFFFFF


def _grid(n, dim):
    m = (torch.arange(n, dtype=torch.float64, device=DEV) + 0.5) / n
    if dim == 1:
        return m[:, None].contiguous()
    return torch.stack([m.repeat(n), m.repeat_interleave(n)], 1).contiguous()


def _test_grid(n, dim):
    t = torch.linspace(0.0, 1.0, n, dtype=torch.float64, device=DEV)
    if dim == 1:
        return t[:, None].contiguous()
    return torch.stack([t.repeat(n), t.repeat_interleave(n)], 1).contiguous()


def _row_sets(case, seed):
    """The row sets of a case: dicts of points, rhs, c0, c1, c2, weight."""
    g = _generator(seed)
    n, dim = case["n"], case["dim"]
    zero = (0.0, 0.0)
    if case["pde"] == "oscillator":
        # u'' + 2 beta u' + w^2 u = 0, u(0) and u'(0) given, w = 80
        w, beta = 80.0, 16.0
        t = (torch.arange(1, n + 1, dtype=torch.float64, device=DEV) / n)[:, None].contiguous()
        z = torch.zeros((1, 1), dtype=torch.float64, device=DEV)
        start = torch.rand(2, generator=g, dtype=torch.float64, device=DEV) + 0.5
        return [dict(points=t, rhs=torch.zeros(n, dtype=torch.float64, device=DEV), c0=w * w,
                     c1=(2 * beta, 0.0), c2=(1.0, 0.0)),
                dict(points=z, rhs=start[:1].clone(), c0=1.0, weight=w ** 4),
                dict(points=z.clone(), rhs=start[1:] * w, c1=(1.0, 0.0), weight=w ** 2)]
    # -Laplace u = f, u = 0 on the boundary: a random sum of sine modes
    modes, kmax = 8, 32
    x = _grid(n, dim)
    k = torch.randint(1, kmax + 1, (modes, dim), generator=g, device=DEV).double()
    A = torch.randn(modes, generator=g, dtype=torch.float64, device=DEV)
    f = torch.zeros(x.shape[0], dtype=torch.float64, device=DEV)
    for m in range(modes):
        s = torch.full_like(f, 1.0) * A[m]
        for i in range(dim):
            s = s * torch.sin(math.pi * k[m, i] * x[:, i])
        f += s
    if dim == 1:
        b = torch.tensor([[0.0], [1.0]], dtype=torch.float64, device=DEV)
    else:
        m = (torch.arange(n, dtype=torch.float64, device=DEV) + 0.5) / n
        z, o = torch.zeros_like(m), torch.ones_like(m)
        b = torch.cat([torch.stack(p, 1) for p in ((m, z), (o, m), (m.flip(0), o), (z, m.flip(0)))])
    return [dict(points=x, rhs=f, c2=(-1.0, -1.0 if dim == 2 else 0.0)),
            dict(points=b.contiguous(), rhs=torch.zeros(b.shape[0], dtype=torch.float64, device=DEV),
                 c0=1.0, weight=(kmax * math.pi) ** 4)]


def _solver(case, seed, precision):
    d = case["dim"]
    return E.Solver(d, (0.0,) * d, (1.0,) * d, _levels(case), _delta(case), case["K"],
                    seed=_model_seed(seed), precision=PREC[precision])


def _eval_inputs(case, seed):
    g = _generator(seed)
    x = torch.rand((case["points"], case["dim"]), generator=g, dtype=torch.float64, device=DEV)
    a = torch.randn(_subdomains(case) * case["K"], generator=g, dtype=torch.float64, device=DEV)
    return x, a


def _gram_pairs(case, seed):
    """48 subdomain pairs: at 8 places of the finest level, the subdomain with
    itself, with neighbours and with the coarser levels' subdomains over it."""
    lev, r = _levels(case), np.random.default_rng(seed)
    off = np.concatenate([[0], np.cumsum([v * v for v in lev])])
    n, out = lev[-1], []
    for _ in range(8):
        ix, iy = (int(v) for v in r.integers(0, n, 2))
        s = int(off[-2]) + iy * n + ix
        out.append((s, s))
        if ix + 1 < n:
            out.append((s, s + 1))
        if iy + 1 < n:
            out.append((s, s + n))
        for l, v in enumerate(lev[:-1]):
            out.append((int(off[l]) + (iy * v // n) * v + ix * v // n, s))
    return np.array(out[:48], dtype=np.int32)


def _network_weights(case, seed):
    K, H = case["K"], 64
    r = np.random.default_rng(seed)
    parts = [r.standard_normal(H * K) / math.sqrt(K), 0.1 * r.standard_normal(H)]
    for _ in range(3):
        parts += [r.standard_normal(H * H) / math.sqrt(H), r.standard_normal(H * H) / math.sqrt(H),
                  0.1 * r.standard_normal(H)]
    parts += [r.standard_normal(K * H) / math.sqrt(H), 0.1 * r.standard_normal(K)]
    return np.concatenate(parts).astype(np.float32)


def _network_inputs(case, seed):
    r = np.random.default_rng([seed, 1])
    shape = (case["batch"], _subdomains(case), case["K"])
    x = r.standard_normal(shape).astype(np.float32)
    t = r.standard_normal(shape).astype(np.float32)
    wb = (0.5 + r.random(case["batch"])).astype(np.float32)
    return x, t, wb


def _batch_sizes(case):
    """Uneven instances: subdomains per dimension, features and grid side, each
    up to the case's, with several points per feature in a support."""
    r = np.random.default_rng([case["instances"], case["n"]])
    out = []
    for _ in range(case["instances"]):
        K = int(r.choice([k for k in (32, 64, 128) if k <= case["K"]]))
        n = int(r.integers(case["n"] // 2, case["n"] + 1))
        cap = min(case["n_sub"], int(2 * n / math.sqrt(4 * K)))
        out.append((int(r.integers(2, max(cap, 2) + 1)), K, n))
    return out


def _batch_problems(case, seed):
    t = np.linspace(0.0, 1.0, 64)
    xt = np.stack([np.tile(t, 64), np.repeat(t, 64)], 1)
    out = []
    for i, (ns, K, n) in enumerate(_batch_sizes(case)):
        c = dict(pde="poisson", dim=2, levels=str(ns), K=K, n=n)
        sets = []
        for s in _row_sets(c, seed * 1009 + i):
            sets.append(types.SimpleNamespace(
                points=s["points"].cpu().numpy(), rhs=s["rhs"].cpu().numpy(), c0=s.get("c0", 0.0),
                c1=(0.0, 0.0), c2=s.get("c2", (0.0, 0.0)), weight=s.get("weight")))
        out.append(types.SimpleNamespace(
            dim=2, lo=(0.0, 0.0), hi=(1.0, 1.0), levels=(ns,), delta=2.0, features=K,
            seed=_model_seed(seed + i), weight_scale=1.0, placement="cell", interior=sets[0],
            boundary=sets[1:], exact=lambda p: np.zeros(p.shape[0]) + 1.0, test_points=xt,
            n_columns=ns * ns * K))
    return out


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind == "eval":
        x, a = _eval_inputs(case, seed)
        st.update(solver=_solver(case, seed, "fp64"), x=x, out=torch.empty_like(x[:, 0]))
        st["solver"].set_coeffs(a.cpu().numpy())
        return st
    if kind == "batch":
        st.update(problems=_batch_problems(case, seed), opts=E.default_solve_opts(
            max_iter=case["iters"], atol=0.0, btol=0.0, shift=case["shift"], check_every=10))
        return st
    sets = _row_sets(case, seed)
    if kind == "fit":
        st.update(sets=sets, seed=seed, x=_test_grid(case["points"], 1))
        st["out"] = torch.empty_like(st["x"][:, 0])
        return st
    s = _solver(case, seed, case["precision"])
    st["solver"] = s
    if kind == "assemble":
        st["sets"] = sets
        return st
    s.assemble(sets)
    if kind in ("solve", "qr"):
        st["x"] = _test_grid(96, 2) if kind == "solve" else _test_grid(case["points"], 1)
        st["out"] = torch.empty_like(st["x"][:, 0])
    elif kind == "gram":
        st["pairs"] = _gram_pairs(case, seed)
        K = case["K"]
        st["out"] = torch.empty((len(st["pairs"]), K, K), dtype=torch.float64, device=DEV)
    elif kind == "network":
        s.gnn_set_weights(_network_weights(case, seed))
        st["inputs"] = _network_inputs(case, seed)
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _plain(iters):
    """The paper's protocol: unpreconditioned LSQR from a cold start."""
    return dict(preconditioner=E.PREC_NONE, max_iter=iters, atol=0.0, btol=0.0, check_every=50)


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "eval":
        return st["solver"].eval(st["x"], st["out"])
    if kind == "fit":
        with _solver(case, st["seed"], case["precision"]) as s:
            s.assemble(st["sets"])
            s.solve(**_plain(case["iters"]))
            u = s.eval(st["x"], st["out"])
            return dict(u=u, coeffs=s.coeffs())
    if kind == "qr":
        # the model and the rank: coefficients at the rank cut are not unique
        s = st["solver"]
        info = s.solve(method=E.SOLVE_QR, rcond=case["rcond"])
        return dict(u=s.eval(st["x"], st["out"]), rank=int(info.rank))
    if kind == "assemble":
        s = st["solver"]
        s.assemble(st["sets"])
        s.solve(**_plain(1))   # the first step: a multiple of M^T h over the whole system
        a = s.coeffs()
        return a if case["precision"] == "fp64" else a.astype(np.float32)
    if kind == "solve":
        s = st["solver"]
        s.solve(max_iter=case["iters"], atol=0.0, btol=0.0, shift=case["shift"], check_every=10)
        return s.eval(st["x"], st["out"]).float()
    if kind == "gram":
        s = st["solver"]
        s.compute_gram()
        p, lib = st["pairs"], E.lib()
        rc = lib.elmfb_get_gram(s.h, len(p), p.ctypes.data, st["out"].data_ptr())
        if rc != E.OK:
            raise E.ElmfbError(rc, lib.elmfb_last_error(s.h).decode())
        return st["out"].float()
    if kind == "batch":
        _, outs, _ = E.batch_solve(st["problems"], precision=E.FP32, n_workers=8, opts=st["opts"])
        return np.concatenate(outs).astype(np.float32)
    x, t, wb = st["inputs"]
    y, grad, loss = st["solver"].gnn_eval(x, t, wb, grad=True)
    return dict(y=y, grad=grad, loss=np.float32(loss))


# ---------------------------------------------------------------------------
# the least work
# ---------------------------------------------------------------------------
def _cover(levels, dim, delta):
    """Mean number of subdomains that cover a point, summed over the levels."""
    total = 0.0
    for n in levels:
        mu = (np.arange(n) + 0.5) / n
        half = 0.5 * delta / n
        total += float(np.sum(np.minimum(mu + half, 1.0) - np.maximum(mu - half, 0.0))) ** dim
    return total


def _system_work(case, iters):
    """Bytes and flops of assembling and `iters` LSQR steps (one read each)."""
    lev, dim, K = _levels(case), case["dim"], case["K"]
    rows = case["n"] ** dim + (4 * case["n"] if dim == 2 else 2)
    nnz = rows * K * _cover(lev, dim, _delta(case))
    size = 4 if case["precision"] in ("fp32", "mixed") else 8
    cols = _subdomains(case) * K
    return dict(rows=rows, nnz=nnz, panel=nnz * size, cols=cols,
                inputs=8.0 * rows * (dim + 1) + 8.0 * cols * (dim + 1),
                step=nnz * size + 16.0 * rows + 40.0 * cols, flops=4.0 * nnz * iters)


def work(case):
    kind = case["kind"]
    if kind == "eval":
        n, dim, K = case["points"], case["dim"], case["K"]
        terms = n * K * _cover(_levels(case), dim, _delta(case))
        cols = _subdomains(case) * K
        return dict(bytes=8.0 * n * (dim + 1) + 8.0 * cols * (dim + 2),
                    flops=terms * (2 * dim + 3))
    if kind == "batch":
        b = f = 0.0
        for ns, K, n in _batch_sizes(case):
            c = dict(dim=2, levels=str(ns), K=K, n=n, precision="fp32")
            w = _system_work(c, case["iters"])
            b += w["inputs"] + w["panel"] * 2 + w["step"] * (case["iters"] + 1)
            f += w["flops"] + w["nnz"] * (K + 12)
        return dict(bytes=b, flops=f)
    if kind == "network":
        n, H, K, B = _subdomains(case), 64, case["K"], case["batch"]
        weights = 2 * K * H + 3 * 2 * H * H + 4 * H + K
        return dict(bytes=4.0 * (3 * B * n * K + 2 * weights),
                    flops=6.0 * B * n * (2 * K * H + 6 * H * H))
    if kind == "fit":
        w = _system_work(case, case["iters"])
        return dict(bytes=w["inputs"] + w["panel"] + w["step"] * (case["iters"] + 1),
                    flops=w["flops"] + w["nnz"] * 12)
    w = _system_work(case, case.get("iters", 1))
    if kind == "qr":
        m, n = w["rows"], w["cols"]
        return dict(bytes=w["panel"] + 8.0 * n, flops=2.0 * m * n * n - 2.0 / 3.0 * n ** 3)
    if kind == "assemble":
        return dict(bytes=w["inputs"] + w["panel"] + 2 * w["step"], flops=w["flops"] + w["nnz"] * 12)
    if kind == "solve":
        return dict(bytes=w["panel"] + w["step"] * (case["iters"] + 1),
                    flops=w["flops"] + w["nnz"] * case["K"])
    # Gram blocks of every pair of subdomains that share points, each once
    c = _cover(_levels(case), case["dim"], _delta(case))
    K = case["K"]
    return dict(bytes=2.0 * w["nnz"], flops=K * (c + 1) * w["nnz"])


# ---------------------------------------------------------------------------
# the same results in 64 bits, by plain torch
# ---------------------------------------------------------------------------
def _parameters(case, seed):
    """Hidden weights and biases: the SplitMix64 stream, uniform in (-1, 1)."""
    dim = case["dim"]
    N = _subdomains(case) * case["K"]
    i = np.arange(1, N * (dim + 1) + 1, dtype=np.uint64)
    with np.errstate(over="ignore"):
        z = np.uint64(_model_seed(seed)) + i * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    v = 2.0 * ((z >> np.uint64(40)).astype(np.float64) * 2.0 ** -24) - 1.0
    v = torch.from_numpy(v).to(DEV).reshape(N, dim + 1)
    return v[:, :dim].contiguous(), v[:, dim].contiguous()


def _level_terms(x, n, delta):
    """Covering subdomains of every point at one level (idx [p, c]), their
    normalised windows with first and second derivatives, and the scaled
    coordinates ([p, c] or [p, c, dim])."""
    p, dim = x.shape
    h = 1.0 / n
    sigma = 0.5 * delta * h
    c1 = int(math.ceil(delta))
    per = []
    for i in range(dim):
        first = torch.ceil(x[:, i] / h - 0.5 - 0.5 * delta)
        j = first[:, None] + torch.arange(c1, device=x.device, dtype=torch.float64)
        dx = x[:, i:i + 1] - (j + 0.5) * h
        inside = (j >= 0) & (j < n) & (dx.abs() < sigma)
        u = (sigma - dx.abs()) / sigma   # cos(theta / 2) = sin(pi u / 2)
        co, si = torch.sin(0.5 * math.pi * u), torch.cos(0.5 * math.pi * u) * torch.sign(dx)
        g = math.pi / sigma
        f = torch.where(inside, 4 * co ** 4, 0.0)
        f1 = torch.where(inside, -8 * co ** 3 * si * g, 0.0)
        f2 = torch.where(inside, 4 * co ** 2 * (3 * si ** 2 - co ** 2) * g * g, 0.0)
        per.append((j.clamp(0, n - 1).long(), dx / sigma, f, f1, f2))
    if dim == 1:
        j, xt, f, f1, f2 = per[0]
        idx, xt, w, dw, ddw = j, xt[:, :, None], f, [f1], [f2]
    else:
        (j0, x0, f0, a0, b0), (j1, x1, f1, a1, b1) = per

        def outer(v1, v0):   # y slower, x faster
            return (v1[:, :, None] * v0[:, None, :]).reshape(p, -1)
        idx = (j1[:, :, None] * n + j0[:, None, :]).reshape(p, -1)
        one = torch.ones_like(x0)
        xt = torch.stack([outer(one, x0), outer(x1, one)], 2)
        w = outer(f1, f0)
        dw, ddw = [outer(f1, a0), outer(a1, f0)], [outer(f1, b0), outer(b1, f0)]
    S = w.sum(1, keepdim=True)
    om, dom, ddom = w / S, [], []
    for i in range(dim):
        dS, ddS = dw[i].sum(1, keepdim=True), ddw[i].sum(1, keepdim=True)
        a = dS / S
        dom.append((dw[i] - w * a) / S)
        ddom.append((ddw[i] - 2 * dw[i] * a - w * ddS / S + 2 * w * a * a) / S)
    return idx, om, dom, ddom, xt, sigma


def _exact_eval(case, seed, x, a):
    W, b = _parameters(case, seed)
    lev, K, dim = _levels(case), case["K"], case["dim"]
    W, b, a = W.reshape(-1, K, dim), b.reshape(-1, K), a.reshape(-1, K)
    out = torch.zeros(x.shape[0], dtype=torch.float64, device=x.device)
    for p in range(0, x.shape[0], 1 << 16):
        xp, off = x[p:p + (1 << 16)], 0
        for n in lev:
            idx, om, _, _, xt, _ = _level_terms(xp, n, _delta(case))
            idx = idx + off
            for c in range(idx.shape[1]):
                s = b[idx[:, c]]
                for i in range(dim):
                    s = s + W[idx[:, c], :, i] * xt[:, c, i:i + 1]
                out[p:p + (1 << 16)] += om[:, c] * (torch.tanh(s) * a[idx[:, c]]).sum(1)
            off += n ** dim
    return out / len(lev)


class _System:
    """M and h in 64 bits: per level the covering subdomains of every row and
    the K entries of each."""

    def __init__(self, case, seed, sets=None):
        W, b = _parameters(case, seed)
        lev, K, dim, L = _levels(case), case["K"], case["dim"], len(_levels(case))
        W, b = W.reshape(-1, K, dim), b.reshape(-1, K)
        sets = _row_sets(case, seed) if sets is None else sets
        self.K, self.nsub, self.off, self.dim = K, _subdomains(case), [], dim
        self.lev = lev
        x, hs, co = [], [], []
        for k, s in enumerate(sets):
            n = s["rhs"].shape[0]
            sc = 1.0 / math.sqrt(n) if k == 0 else math.sqrt(s["weight"] / n)
            x.append(s["points"])
            hs.append(s["rhs"] * sc)
            v = [s.get("c0", 0.0), *s.get("c1", (0.0, 0.0))[:dim], *s.get("c2", (0.0, 0.0))[:dim]]
            co.append((torch.tensor(v, dtype=torch.float64, device=DEV) * (sc / L)).expand(n, -1))
        x, self.h, co = torch.cat(x), torch.cat(hs), torch.cat(co)
        self.idx, self.E = [], []
        off = 0
        for n in lev:
            I, V = [], []
            for p in range(0, x.shape[0], 1 << 17):
                xp, cp = x[p:p + (1 << 17)], co[p:p + (1 << 17)]
                idx, om, dom, ddom, xt, sigma = _level_terms(xp, n, _delta(case))
                idx = idx + off
                A = cp[:, :1] * om
                for i in range(dim):
                    A = A + cp[:, 1 + i:2 + i] * dom[i] + cp[:, 1 + dim + i:2 + dim + i] * ddom[i]
                V1 = torch.empty((*idx.shape, K), dtype=torch.float64, device=DEV)
                for c in range(idx.shape[1]):
                    w = W[idx[:, c]]
                    s = b[idx[:, c]]
                    for i in range(dim):
                        s = s + w[:, :, i] * xt[:, c, i:i + 1]
                    phi = torch.tanh(s)
                    t = 1 - phi * phi
                    v = phi * A[:, c:c + 1]
                    for i in range(dim):
                        be = cp[:, 1 + i] * om[:, c] + 2 * cp[:, 1 + dim + i] * dom[i][:, c]
                        ga = cp[:, 1 + dim + i] * om[:, c]
                        d = w[:, :, i] / sigma
                        v = v + t * (be[:, None] * d - 2 * phi * ga[:, None] * d * d)
                    V1[:, c] = v
                I.append(idx)
                V.append(V1)
            self.idx.append(torch.cat(I))
            self.E.append(torch.cat(V))
            self.off.append(off)
            off += n ** dim

    def mul(self, t):
        t = t.reshape(-1, self.K)
        out = torch.zeros_like(self.h)
        for idx, E_ in zip(self.idx, self.E):
            for c in range(idx.shape[1]):
                out += (E_[:, c] * t[idx[:, c]]).sum(1)
        return out

    def tmul(self, u):
        out = torch.zeros((self.nsub, self.K), dtype=torch.float64, device=DEV)
        for idx, E_ in zip(self.idx, self.E):
            for c in range(idx.shape[1]):
                out.index_add_(0, idx[:, c], E_[:, c] * u[:, None])
        return out.reshape(-1)

    def columns(self, s):
        """Dense columns [rows, K] of subdomain s."""
        l = max(k for k in range(len(self.off)) if self.off[k] <= s)
        return torch.where((self.idx[l] == s)[:, :, None], self.E[l], 0.0).sum(1)

    def factors(self, shift):
        """X_j = L_j^-1 of every shifted diagonal block."""
        G = torch.zeros((self.nsub, self.K, self.K), dtype=torch.float64, device=DEV)
        for idx, E_ in zip(self.idx, self.E):
            live = (E_ != 0).any(2).reshape(-1)
            flat, rows = idx.reshape(-1)[live], E_.reshape(-1, self.K)[live]
            order = torch.argsort(flat, stable=True)
            subs, count = torch.unique_consecutive(flat[order], return_counts=True)
            at = 0
            for s, n in zip(subs.tolist(), count.tolist()):
                r = rows[order[at:at + n]]
                G[s] = r.T @ r
                at += n
        tr = G.diagonal(dim1=1, dim2=2).sum(1)
        eye = torch.eye(self.K, dtype=torch.float64, device=DEV)
        L = torch.linalg.cholesky(G + (shift * tr / self.K)[:, None, None] * eye)
        return torch.linalg.solve_triangular(L, eye.expand_as(L), upper=False)

    def dense(self):
        M = torch.zeros((self.h.shape[0], self.nsub, self.K), dtype=torch.float64, device=DEV)
        r = torch.arange(self.h.shape[0], device=DEV)
        for idx, E_ in zip(self.idx, self.E):
            for c in range(idx.shape[1]):
                M.index_put_((r, idx[:, c]), E_[:, c], accumulate=True)
        return M.reshape(self.h.shape[0], -1)


def _exact_lsqr(S, iters, X=None):
    """Coefficients after `iters` steps of LSQR (Paige & Saunders 1982) on M P,
    P = X^T per subdomain (identity without X)."""
    K = S.K

    def P(y):
        return y if X is None else torch.einsum("sik,si->sk", X, y.reshape(-1, K)).reshape(-1)

    def Pt(z):
        return z if X is None else torch.einsum("sik,sk->si", X, z.reshape(-1, K)).reshape(-1)
    beta = S.h.norm()
    u = S.h / beta
    v = Pt(S.tmul(u))
    alpha = v.norm()
    v = v / alpha
    w, y = v.clone(), torch.zeros_like(v)
    phib, rhob = beta, alpha
    for _ in range(iters):
        u = S.mul(P(v)) - alpha * u
        beta = u.norm()
        u = u / beta
        v = Pt(S.tmul(u)) - beta * v
        alpha = v.norm()
        v = v / alpha
        rho = torch.sqrt(rhob * rhob + beta * beta)
        c, s = rhob / rho, beta / rho
        theta, rhob = s * alpha, -c * alpha
        phi, phib = c * phib, s * phib
        y = y + (phi / rho) * w
        w = v - (theta / rho) * w
    return P(y)


def _exact_network(case, seed):
    S = _System(case, seed)
    n, K, H = S.nsub, case["K"], 64
    on = torch.zeros((S.h.shape[0], n), dtype=torch.float32, device=DEV)
    r = torch.arange(S.h.shape[0], device=DEV)
    for idx, E_ in zip(S.idx, S.E):
        for c in range(idx.shape[1]):
            live = (E_[:, c] != 0).any(1)
            on[r[live], idx[live, c]] = 1.0
    adj = ((on.T @ on) > 0).double()
    adj.fill_diagonal_(0.0)
    mean = adj / adj.sum(1, keepdim=True).clamp(min=1.0)
    w = torch.from_numpy(_network_weights(case, seed)).to(DEV).double().requires_grad_(True)
    x, t, wb = (torch.from_numpy(v).to(DEV).double() for v in _network_inputs(case, seed))
    o = 0

    def take(*shape):
        nonlocal o
        k = int(np.prod(shape))
        o += k
        return w[o - k:o].reshape(shape)
    a = torch.relu(x @ take(H, K).T + take(H))
    for _ in range(3):
        ws, wn, b = take(H, H), take(H, H), take(H)
        a = torch.relu(a @ ws.T + torch.einsum("st,btk->bsk", mean, a) @ wn.T + b)
    y = a @ take(K, H).T + take(K)
    loss = (wb * ((y - t) ** 2).sum((1, 2))).mean()
    loss.backward()
    return dict(y=y.detach(), grad=w.grad, loss=loss.detach())


def exact(case, seed):
    kind = case["kind"]
    if kind == "eval":
        return _exact_eval(case, seed, *_eval_inputs(case, seed))
    if kind == "fit":
        a = _exact_lsqr(_System(case, seed), case["iters"])
        return dict(u=_exact_eval(case, seed, _test_grid(case["points"], 1), a), coeffs=a)
    if kind == "assemble":
        return _exact_lsqr(_System(case, seed), 1)
    if kind == "solve":
        S = _System(case, seed)
        a = _exact_lsqr(S, case["iters"], S.factors(case["shift"]))
        return _exact_eval(case, seed, _test_grid(96, 2), a)
    if kind == "gram":
        S = _System(case, seed)
        return torch.stack([S.columns(i).T @ S.columns(j) for i, j in _gram_pairs(case, seed)])
    if kind == "batch":
        out = []
        for i, (ns, K, n) in enumerate(_batch_sizes(case)):
            c = dict(pde="poisson", dim=2, levels=str(ns), K=K, n=n)
            S = _System(c, seed + i, _row_sets(c, seed * 1009 + i))
            a = _exact_lsqr(S, case["iters"], S.factors(case["shift"]))
            out.append(_exact_eval(c, seed + i, _test_grid(64, 2), a))
        return torch.cat(out)
    if kind == "network":
        return _exact_network(case, seed)
    # qr: the truncated least-squares solution by singular values
    S = _System(case, seed)
    a = np.linalg.lstsq(S.dense().cpu().numpy(), S.h.cpu().numpy(), rcond=case["rcond"])[0]
    a = torch.from_numpy(a).to(DEV)
    return dict(u=_exact_eval(case, seed, _test_grid(case["points"], 1), a), rank=None)
