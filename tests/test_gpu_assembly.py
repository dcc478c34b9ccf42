"""GPU parity of create (parameters) and assembly (M, h) against the FP64 oracle.

Tolerance on entries (paper §3 entries; precision reading): |M_gpu - M_oracle|
<= tol * max(T, 1e-3 S), with T the largest magnitude sum of product-rule and
quotient-rule terms over the K features of the same row and subdomain block
(the oracle's ``bound``), S the largest T of that subdomain block over all
rows, tol = 1e-12 for FP64 and DF32 (FP32 pair) panels and 1e-6 for FP32
panels.  The 1e-3 S floor
covers points within rounding distance of a support edge, where the window and
its derivatives vanish and an entry's relative value is not determined by the
FP64 coordinates.
"""
import numpy as np
import pytest

import paper_2409_01949_gb300 as E
import workloads as WL
from oracle import decomposition as OD
from oracle import rng as OR
from oracle import system as OS

pytestmark = pytest.mark.gpu

TOL = {E.FP64: 1e-12, E.FP32: 1e-6, E.MIXED: 1e-6, E.DF32: 1e-12}

SMALL = {
    "poisson1d_full": (WL.config_poisson1d, [E.FP64, E.FP32, E.DF32]),
    "dho_L1-8_K24": (lambda: WL.dho(levels=(1, 2, 4, 8), features=24, n_interior=1000),
                     [E.FP64, E.FP32, E.DF32]),
    "poisson2d_L1-4_K64": (lambda: WL.poisson2d(levels=(1, 2, 4), features=64, n_side=60,
                                                n_boundary_side=60),
                           [E.FP64, E.FP32, E.MIXED, E.DF32]),
    "dho_paper_K12_delta2.9_endpoint": (WL.dho_paper_baseline, [E.FP64]),
    "poisson2d_delta2.9_K40": (lambda: WL.poisson2d(levels=(3, 5), features=40, n_side=50,
                                                    n_boundary_side=50, delta=2.9), [E.FP32]),
    "poisson2d_ragged_K33": (lambda: WL.poisson2d(levels=(1, 3, 7), features=33, n_side=37,
                                                  n_boundary_side=11),
                            [E.FP64, E.FP32, E.DF32]),
    # §4.4: the L-shaped domain, subdomains of the cut-out square discarded
    "helmholtz_L_w8_J16_K16": (WL.helmholtz_lshape, [E.FP64, E.FP32, E.DF32]),
    "helmholtz_L_J1-8-16_K12_endpoint": (
        lambda: WL.helmholtz_lshape(levels=(1, 8, 16), features=12, n_grid=40, n_long=40,
                                    n_short=20, placement="endpoint"), [E.FP64, E.DF32]),
    # the largest feature counts: K = 256 (the library's maximum), K = 160 (past
    # the fused pass's 128, ragged against 32-lane slices)
    "poisson1d_Kmax256": (lambda: WL.poisson1d(levels=(2, 4), features=256, n_interior=90),
                          [E.FP64, E.FP32, E.DF32]),
    "poisson2d_K160": (lambda: WL.poisson2d(levels=(2,), features=160, n_side=26,
                                            n_boundary_side=9), [E.FP64, E.FP32]),
    # §4.3: the hard-constraint ansatz, no boundary rows
    "laplace_n4_J16_K16": (WL.laplace_multiscale, [E.FP64, E.FP32, E.DF32]),
    "laplace_n2_J1-4-8_K20_ansatz": (
        lambda: WL.laplace_multiscale(omegas=(3, 5), levels=(1, 4, 8), features=20, n_grid=30,
                                      delta=2.0), [E.FP64, E.FP32]),
}


def _scale(bound, K):
    T = OS.block_max(bound, K)
    S = T.max(axis=0, keepdims=True)
    return np.maximum(T, 1e-3 * S)


def _compare(P, prec, rows=None):
    with E.Solver.from_problem(P, precision=prec) as s:
        s.assemble_problem(P)
        sz = s.sizes()
        rows = np.arange(P.n_rows) if rows is None else np.asarray(rows)
        Mg, hg = s.get_rows(rows)
        ref = OS.assemble(P, rows=rows, fmt="dense", with_bound=True)
        scale = _scale(ref["bound"], P.features)
        err = np.abs(Mg - ref["M"])
        ratio = float((err / np.maximum(scale, 1e-300)).max())
        assert np.all(err <= TOL[prec] * scale), f"max err/scale = {ratio:.3e}"
        assert np.allclose(hg, ref["h"], rtol=1e-15, atol=0)
        return sz, ratio


@pytest.mark.parametrize("name", list(SMALL))
def test_assembly_all_rows(name):
    make, precs = SMALL[name]
    P = make()
    for prec in precs:
        sz, ratio = _compare(P, prec)
        assert sz.n_rows == P.n_rows and sz.n_columns == OD.n_columns(P)


def test_stored_entry_count_matches_closed_form():
    """1D Poisson, 16 cell-centred subdomains, delta = 2, 2000 midpoints, K = 64.

    The oracle's nonzeros are 3862 row-subdomain pairs (247168 entries).  The
    panels also store, as exact zeros, the 15 centre points mu_0..mu_14 that
    lie on the left edge of the open support of their right neighbour (they
    share that neighbour's cell): 3877 * 64 = 248128 stored entries.
    """
    P = WL.config_poisson1d()
    with E.Solver.from_problem(P, precision=E.FP64) as s:
        s.assemble_problem(P)
        assert s.sizes().nnz == 248128


def test_parameters_bitwise_equal_to_oracle_stream():
    P = WL.poisson2d(levels=(1, 2, 4), features=16, n_side=8)
    with E.Solver.from_problem(P) as s:
        W, b = s.params()
    Wo, bo = OR.draw_parameters(P.seed, P.n_columns, 2, P.weight_scale)
    assert np.array_equal(W, Wo) and np.array_equal(b, bo)


def test_discarded_subdomains_keep_their_parameter_draws():
    """With holes the kept columns carry the draws of their full-grid columns
    (the oracle's stream restricted to the kept subdomains)."""
    P = WL.helmholtz_lshape(levels=(1, 4, 8), features=8)
    levels = OD.build_levels(2, P.lo, P.hi, P.levels, P.delta, P.features, P.placement, P.holes)
    full = np.concatenate([lev.param_offset + np.arange(lev.n_sub * P.features)
                           .reshape(lev.n_sub, P.features)[lev.keep].ravel() for lev in levels])
    with E.Solver.from_problem(P) as s:
        W, b = s.params()
        assert s.sizes().n_subdomains == sum(int(l.keep.sum()) for l in levels)
    Wo, bo = OR.draw_parameters(P.seed, P.n_columns_full, 2, P.weight_scale)
    assert np.array_equal(W, Wo[full]) and np.array_equal(b, bo[full])


@pytest.mark.parametrize("maker,prec", [(WL.config_poisson2d_ml, E.FP32),
                                        (WL.config_dho_ml, E.FP32),
                                        (WL.config_poisson2d_large, E.FP32)])
def test_assembly_full_size_sampled_rows(maker, prec):
    """Full workload sizes, as assembled for the benchmark; rows sampled for the oracle."""
    P = maker()
    rng = np.random.default_rng(7)
    NI = P.interior.points.shape[0]
    rows = np.unique(np.concatenate([rng.choice(NI, 200, replace=False), [0, NI - 1],
                                     NI + rng.choice(P.n_rows - NI, min(32, P.n_rows - NI),
                                                     replace=False)]))
    _compare(P, prec, rows)


def test_out_of_box_point_rejected():
    P = WL.poisson1d(levels=(4,), features=8, n_interior=20)
    pts = P.interior.points.copy()
    pts[3, 0] = 1.5
    with E.Solver.from_problem(P) as s:
        with pytest.raises(E.ElmfbError) as ei:
            s.assemble([dict(points=pts, rhs=P.interior.rhs, c2=(-1.0,))])
        assert ei.value.code == E.ERR_INVALID_ARG


def test_invalid_config_rejected():
    with pytest.raises(E.ElmfbError) as ei:
        E.Solver(1, (0.0,), (1.0,), (4,), delta=1.0, features=8)
    assert ei.value.code == E.ERR_INVALID_ARG


def test_empty_boundary_set_and_boundary_points():
    """A boundary set with zero points is allowed; points on the box edge are inside."""
    P = WL.poisson1d(levels=(2, 4), features=8, n_interior=30)
    sets = [dict(points=P.interior.points, rhs=P.interior.rhs, c2=(-1.0,)),
            dict(points=np.zeros((0, 1)), rhs=np.zeros(0), c0=1.0, weight=1.0, n=0),
            dict(points=np.array([[0.0], [1.0]]), rhs=np.zeros(2), c0=1.0, weight=4.0)]
    with E.Solver.from_problem(P) as s:
        s.assemble(sets)
        assert s.sizes().n_rows == 32


# weight scales at and past the ends of the fixed-point range (1/16 .. 1), a
# scale that is no power of two, K at the edges of the 64-feature passes, one
# axis and two
@pytest.mark.parametrize("dim,K,a", [(1, 1, 1.0), (1, 32, 1.0 / 16), (1, 65, 0.7), (1, 96, 0.05),
                                     (2, 31, 1.0), (2, 64, 0.06), (2, 100, 0.3), (2, 8, 1.5)])
@pytest.mark.parametrize("prec", [E.FP64, E.DF32])
def test_entries_over_weight_scales(dim, K, a, prec):
    """FP64 entries and FP32 pairs against the oracle at 100 times the FP64
    unit (48-bit pairs: 2^-48) of the block's term scale: the arithmetic after
    the windows is a dozen roundings, the windows' second derivatives lose two
    digits at most to the quotient rule's cancellation."""
    mk = WL.poisson1d if dim == 1 else WL.poisson2d
    kw = dict(n_interior=150) if dim == 1 else dict(n_side=20, n_boundary_side=9)
    P = mk(levels=(1, 3, 4), features=K, weight_scale=a, delta=2.3, **kw)
    with E.Solver.from_problem(P, precision=prec) as s:
        s.assemble_problem(P)
        M, _ = s.get_rows(np.arange(P.n_rows))
    ref = OS.assemble(P, fmt="dense", with_bound=True)
    tol = 100 * 2.0 ** -53 if prec == E.FP64 else 2.0 ** -48 + 100 * 2.0 ** -53
    assert np.all(np.abs(M - ref["M"]) <= tol * _scale(ref["bound"], K))


@pytest.mark.parametrize("c", [1e-290, 1e-150, 1.0, 1e150, 1e290])
def test_entries_scale_with_the_operator(c):
    """Entries are linear in the operator's coefficients: rows of terms far
    outside the fixed-point exponents (1e-290, 1e290) go through FP64 and agree
    with the scaled entries of the unscaled operator to a few roundings."""
    P = WL.poisson1d(levels=(2, 5), features=40, n_interior=64)
    out = []
    for k in (1.0, c):
        with E.Solver.from_problem(P, precision=E.FP64) as s:
            s.assemble([dict(points=P.interior.points, rhs=P.interior.rhs, c0=0.5 * k,
                             c1=(0.25 * k, 0.0), c2=(-k, 0.0))])
            out.append(s.get_rows(np.arange(64))[0])
    # 64 ulp of each row's largest entry: the two sides may round in different forms
    top = np.abs(out[0]).max(axis=1, keepdims=True)
    assert np.all(np.abs(out[1] / c - out[0]) <= 64 * 2.0 ** -53 * top)


def test_nonfinite_operator_gives_nonfinite_entries():
    P = WL.poisson1d(levels=(4,), features=12, n_interior=30)
    for bad in (np.inf, np.nan):
        with E.Solver.from_problem(P, precision=E.FP64) as s:
            s.assemble([dict(points=P.interior.points, rhs=P.interior.rhs, c0=bad, c2=(-1.0, 0.0))])
            M, _ = s.get_rows(np.arange(30))
        inside = np.abs((np.arange(4) + 0.5) / 4 - P.interior.points) < 0.25
        assert not np.isfinite(M.reshape(30, 4, 12)[inside]).any()


# operators of one or two terms: with one subdomain over every point the window is
# 1, and an entry is t (c1 w / sigma - 2 phi c2 (w / sigma)^2) + phi c0 alone, which
# goes with a feature's weights to zero
@pytest.mark.parametrize("dim,c0,c1,c2", [
    (1, 0.0, (0.0, 0.0), (-1.0, 0.0)), (1, 0.0, (1.0, 0.0), (0.0, 0.0)),
    (1, 0.0, (2.0 ** -9, 0.0), (1.0, 0.0)), (1, 2.0 ** -12, (0.0, 0.0), (-1.0, 0.0)),
    (2, 0.0, (0.0, 0.0), (-1.0, -1.0)), (2, 0.0, (0.0, 0.0), (1.0, 0.0)),
    (2, 0.0, (0.0, 1.0), (0.0, 0.0)), (2, 0.0, (1.0, 0.0), (0.0, -(2.0 ** 10)))])
@pytest.mark.parametrize("a", [1.0, 0.3, 0.07])
def test_entries_of_small_weights_to_their_own_last_place(dim, c0, c1, c2, a):
    """Every entry against extended precision, relative to its own terms T and what
    its argument's rounding does to them, T + |d entry / d s| (|w x| + |b|): 8 units
    2^-53 of that for the dozen roundings of an FP64 evaluation from exact windows
    (here 1, with derivatives 0).  Arguments whose own terms are below 2^-6 are
    left out: phi is held to 2^-60, not to its last place."""
    Q = np.longdouble
    n, K = 64, 192
    r = np.random.default_rng(5)
    x = r.integers(1, 2 ** 20, (n, dim)) * 2.0 ** -20
    with E.Solver(dim, (0.0,) * dim, (1.0,) * dim, (1,), 2.0, K, seed=11, weight_scale=a,
                  precision=E.FP64) as s:
        W, b = s.params()
        s.assemble([dict(points=x, rhs=np.zeros(n), c0=c0, c1=c1, c2=c2)])
        M, _ = s.get_rows(np.arange(n))
    assert np.abs(W).min() < 2.0 ** -5 * a
    xt = (x - 0.5).astype(Q)            # mu = 1/2, sigma = 1
    W, b = W.reshape(K, dim).astype(Q), b.astype(Q)
    arg = xt @ W.T + b
    terms = np.abs(xt) @ np.abs(W).T + np.abs(b)
    phi = np.tanh(arg)
    t = 1 - phi * phi
    B, C, aB, aC = 0, 0, 0, 0
    for i in range(dim):
        B, aB = B + c1[i] * W[:, i], aB + np.abs(c1[i] * W[:, i])
        C, aC = C + 2 * c2[i] * W[:, i] ** 2, aC + 2 * np.abs(c2[i]) * W[:, i] ** 2
    want = (c0 * phi + t * (B - phi * C)) / 8       # row scale 1 / sqrt(64)
    T = np.abs(c0 * phi) + t * aB + t * np.abs(phi) * aC
    slope = t * abs(c0) + 2 * np.abs(phi) * t * aB + t * np.abs(1 - 3 * phi * phi) * aC
    bound = 8 * Q(2) ** -53 * (T + slope * terms) / 8
    assert np.all((np.abs(M - want) <= bound) | (terms < 2.0 ** -6))
