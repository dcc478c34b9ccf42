"""Model evaluation: the fixed-point kernel and the FP64 one it replaces where
a point's covering subdomains fit a warp and the weight scale is in range.

Tolerance, against the oracle's FP64 evaluation: the windows of a level sum to
1 and |tanh| <= 1, so the terms of u_hat add up to at most S = max_j ||a_j||_1
per level; either side rounds the argument (dim + 1 terms of at most the
weight scale a, plus the scaled coordinate, whose centre subtraction carries
2^-53 / sigma <= 2^-53 n / 1 of the box) and a few products, 16 of them in all:
|difference| <= 16 2^-53 S (1 + (dim + 1) a n_max).
"""
import ctypes as C

import numpy as np
import pytest

import paper_2409_01949_gb300 as E
import workloads as WL
from oracle import evaluate as OE

pytestmark = pytest.mark.gpu


def _problem(dim, levels, K, scale, **kw):
    f = WL.poisson1d if dim == 1 else WL.poisson2d
    return f(levels=levels, features=K, weight_scale=scale, **kw)


def _points(P, n, seed=3):
    """Random points, then support edges, centres and corners."""
    r = np.random.default_rng(seed)
    x = r.random((n, P.dim))
    nl = P.levels[-1]
    special = np.array([0.0, 1.0, 0.5, 0.5 / nl, 1.5 / nl, 1.0 / nl, 1.0 - 0.5 / nl])
    m = min(n, special.size)
    x[:m, 0] = np.clip(special[:m], 0.0, 1.0)
    return x


def _tol(P, a):
    S = np.abs(a).reshape(-1, P.features).sum(axis=1).max()
    return 16 * 2.0 ** -53 * S * (1 + (P.dim + 1) * P.weight_scale * max(P.levels))


# weight scales: 1/16 and 2^16 are the ends of the fixed-point range, 0.06 and
# 70000 just outside it (FP64), 0.3 and 5 not powers of two; K past 32 and
# multiples of it; 40 covering subdomains (delta = 2.9, five levels of nine)
# do not fit a warp
@pytest.mark.parametrize("dim,levels,K,scale,delta,n", [
    (1, (1,), 1, 1.0, 2.0, 1), (1, (16,), 64, 1.0, 2.0, 1000), (1, (1, 2, 4, 8), 33, 0.3, 2.9, 77),
    (1, (5,), 256, 1.0 / 16, 1.5, 9), (1, (8,), 32, 0.06, 2.0, 50), (1, (8,), 40, 5.0, 2.0, 50),
    (1, (4,), 16, 65536.0, 2.0, 200), (1, (4,), 16, 70000.0, 2.0, 50),
    (2, (1, 2, 4), 128, 1.0, 2.0, 333), (2, (3,), 100, 2.0, 2.9, 64), (2, (1, 2, 4, 8, 16), 31, 1.0, 2.0, 2500),
    (2, (3, 4, 5, 6, 7), 8, 1.0, 2.9, 40),
])
def test_eval_matches_oracle(dim, levels, K, scale, delta, n):
    P = _problem(dim, levels, K, scale, delta=delta)
    rng = np.random.default_rng(1)
    a = rng.standard_normal(P.n_columns) * 10.0 ** rng.uniform(-3, 3, P.n_columns)
    X = _points(P, n)
    with E.Solver.from_problem(P) as s:
        s.set_coeffs(a)
        u = s.eval(X)
    assert np.abs(u - OE.u_hat(P, a, X)).max() <= _tol(P, a)


def test_coefficients_outside_the_fixed_point_range():
    """A subdomain whose coefficients are too large for a shared exponent, or
    not finite, is evaluated in FP64: points it does not cover keep their
    values, points it covers see what FP64 gives."""
    P = _problem(1, (8,), 32, 1.0)
    rng = np.random.default_rng(2)
    a = rng.standard_normal(P.n_columns)
    X = np.linspace(0.01, 0.99, 57)[:, None]
    ref = OE.u_hat(P, a, X)
    with E.Solver.from_problem(P) as s:
        for v in (1e300, 1e-300, np.inf, np.nan):
            b = a.copy()
            b[5 * 32 + 3] = v           # subdomain 5 covers (4.5/8, 6.5/8)
            s.set_coeffs(b)
            u = s.eval(X)
            inside = np.abs(X[:, 0] - 5.5 / 8) < 1.0 / 8
            assert np.abs(u[~inside] - ref[~inside]).max() <= _tol(P, a)
            if np.isfinite(v):
                assert np.abs(u - OE.u_hat(P, b, X)).max() <= _tol(P, b)
            else:
                assert not np.isfinite(u[inside]).any()
        s.set_coeffs(np.zeros_like(a))
        assert np.all(s.eval(X) == 0.0)
        # a subdomain of zeros sets no exponent for neighbours of tiny coefficients
        b = 1e-40 * a
        b[5 * 32:6 * 32] = 0.0
        s.set_coeffs(b)
        assert np.abs(s.eval(X) - OE.u_hat(P, b, X)).max() <= _tol(P, b)


def test_points_and_results_in_place_overlapping_or_unaligned():
    """Device buffers are used where they are; overlapping ones and ones not
    aligned to doubles are staged.  All give the values of host arrays."""
    import torch
    P = _problem(1, (4, 8), 24, 1.0)
    a = np.random.default_rng(4).standard_normal(P.n_columns)
    X = _points(P, 301)
    with E.Solver.from_problem(P) as s:
        s.set_coeffs(a)
        ref = s.eval(X)
        x = torch.from_numpy(X).cuda()
        assert np.array_equal(s.eval(x, torch.empty(301, dtype=torch.float64, device="cuda")).cpu().numpy(), ref)
        buf = torch.zeros(302, dtype=torch.float64, device="cuda")
        buf[:301] = x[:, 0]
        torch.cuda.synchronize()
        L = E.lib()
        assert L.elmfb_eval(s.h, C.c_void_p(buf.data_ptr()), 301, C.c_void_p(buf.data_ptr() + 8)) == E.OK
        assert np.array_equal(buf[1:].cpu().numpy(), ref)
        raw = torch.zeros(301 * 8 + 4, dtype=torch.uint8, device="cuda")
        assert L.elmfb_eval(s.h, C.c_void_p(x.data_ptr()), 301, C.c_void_p(raw.data_ptr() + 4)) == E.OK
        assert np.array_equal(raw[4:].cpu().numpy().tobytes(), ref.tobytes())


@pytest.mark.parametrize("levels,K,delta", [((16,), 64, 2.0), ((1, 2, 4, 8), 33, 2.9)])
def test_evaluation_has_no_bias(levels, K, delta):
    """The mean error over 512 points against extended precision.  A point's error
    is about 2e-16 of the model's size (the windows' part of it, independent from
    point to point), so that of the mean is about 1e-17: 2^-54 is five of those.
    Sums whose terms are all rounded to the same side lie above 1e-16."""
    Q = np.longdouble
    P = WL.poisson1d(levels=levels, features=K, n_interior=50, delta=delta)
    r = np.random.default_rng(9)
    a, x = r.standard_normal(P.n_columns), r.random(512)
    with E.Solver.from_problem(P) as s:
        s.set_coeffs(a)
        W, b = s.params()
        u = s.eval(x[:, None])
    W, b, c, t = W.reshape(-1, K).astype(Q), b.reshape(-1, K).astype(Q), a.reshape(-1, K), 0
    pi, off = 2 * np.arccos(Q(0)), 0
    for n in levels:
        d = (x.astype(Q)[:, None] - (np.arange(n) + Q(1) / 2) / n) * n / (Q(delta) / 2)
        w = np.where(np.abs(d) < 1, np.sin(pi / 2 * (1 - np.minimum(np.abs(d), 1))) ** 4, 0)
        w = w / w.sum(axis=1, keepdims=True)
        for j in range(n):
            t = t + w[:, j] * (np.tanh(d[:, j:j + 1] * W[off + j] + b[off + j]) @ c[off + j].astype(Q))
        off += n
    t = t / len(levels)
    assert abs(np.mean(u - t)) <= 2.0 ** -54 * np.sqrt(np.mean(t * t))


@pytest.mark.parametrize("n,launches", [(1, 1), (4, 1), (5, 2), (300, 2)])
def test_few_points_of_a_model_of_many_columns(n, launches):
    """Up to four points of a model of 128^2 subdomains are evaluated in FP64 (one
    launch), which reads their own columns; from five on the columns are packed
    first.  Both agree with the oracle."""
    P = _problem(2, (128,), 8, 1.0, n_side=8, n_boundary_side=4)
    a = np.random.default_rng(6).standard_normal(P.n_columns)
    X = _points(P, n)
    with E.Solver.from_problem(P) as s:
        s.set_coeffs(a)
        before = s.kernel_launches()
        u = s.eval(X)
        assert s.kernel_launches() - before == launches
    assert np.abs(u - OE.u_hat(P, a, X)).max() <= _tol(P, a)


def test_evaluation_on_a_full_device():
    """A model of 8.4 million columns: its packed columns take 270 MB.  With less
    than that free the points are evaluated in FP64, which takes no memory of its
    own, to the same values within the tolerance."""
    import torch
    P = _problem(2, (256,), 128, 1.0, n_side=8, n_boundary_side=4)
    a = np.random.default_rng(8).standard_normal(P.n_columns)
    x = torch.from_numpy(_points(P, 5000)).cuda()
    out = torch.empty((2, 5000), dtype=torch.float64, device="cuda")
    fill = None
    for k in range(2):
        with E.Solver.from_problem(P) as s:
            s.set_coeffs(a)
            torch.cuda.synchronize()
            if k:
                E.trim_memory()
                torch.cuda.empty_cache()
                fill = torch.empty(torch.cuda.mem_get_info()[0] - (160 << 20), dtype=torch.uint8,
                                   device="cuda")
            before = s.kernel_launches()
            s.eval(x, out[k])
            assert s.kernel_launches() - before == (1 if k else 2)
            del fill
            fill = None
        E.trim_memory()
    torch.cuda.empty_cache()
    assert float((out[0] - out[1]).abs().max()) <= 2 * _tol(P, a)


@pytest.mark.parametrize("K", [1, 32, 33, 64, 65, 96, 97, 128, 129, 160, 255, 256])
@pytest.mark.parametrize("dim,levels,delta", [(1, (5,), 2.0), (1, (1, 2, 4, 8, 16, 32), 2.9),
                                              (2, (1, 2, 4), 2.9)])
def test_sums_of_largest_terms(K, dim, levels, delta):
    """Every term at its largest and of one sign: the coefficients just below a
    power of two, with the sign of their features, which a weight scale of 64
    saturates nearly everywhere.  A lane's sums and those over the covering
    subdomains come as close to their bounds as they can."""
    P = _problem(dim, levels, K, 64.0, delta=delta)
    X = np.random.default_rng(2).random((400, dim))
    with E.Solver.from_problem(P) as s:
        _, b = s.params()
        a = np.nextafter(2.0, 0.0) * np.sign(b)
        for v in (a, -a, np.abs(a)):
            s.set_coeffs(v)
            assert np.abs(s.eval(X) - OE.u_hat(P, v, X)).max() <= _tol(P, v)
