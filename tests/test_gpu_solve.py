"""GPU parity of the least-squares solve, model evaluation and error norms.

Solution parity against the oracle's least-squares minimiser (Eq.
multilevel_ls), wherever the dense system fits the oracle's memory: the GPU's
column-pivoted QR solve (ELMFB_SOLVE_QR, the oracle's algorithm) must reach
a relative L2 error against the closed-form solution of at most 1.01x the
oracle's QR error, where that error is taken as the largest over the oracle's
QR of the system in its own row order and in three shuffled row orders (row
order changes no minimiser, only the FP64 rounding; two valid FP64 QRs of the
1-D Poisson system differ by 5% in this error).

The LSQR path (the paper's solver, §3 and §4.1) is held to the paper's own
protocol: at most 1.01x the error of SciPy LSQR from zero run for the full
15000-iteration budget; its iterates are compared with SciPy's.  The QR
minimiser is out of reach of LSQR at these condition numbers (1e17 and
more): it uses singular directions that the Krylov iteration resolves only
after far more than 15000 steps.
"""
import json
import os

import numpy as np
import pytest
import scipy.sparse.linalg as spla

import paper_2409_01949_gb300 as E
import workloads as WL
from oracle import evaluate as OE
from oracle import system as OS

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(__file__), "golden", "oracle_errors.json")


def _golden(name):
    if not os.path.exists(GOLDEN):
        pytest.skip("oracle_errors.json not generated")
    g = json.load(open(GOLDEN))
    if name not in g:
        pytest.skip(f"{name} not in oracle_errors.json")
    return g[name]


def test_plain_lsqr_iterates_match_oracle_lsqr():
    """Without a preconditioner the GPU runs the paper's LSQR; its k-th iterate
    matches SciPy's k-th iterate.  Only the first iterates are comparable: the
    Lanczos bidiagonalisation amplifies rounding, so that a 1e-15 relative
    perturbation of M already moves the 10th iterate by ~20% on this system
    (condition number ~8e3) in any implementation."""
    P = WL.poisson1d(levels=(4,), features=4, n_interior=200, lam=100.0)
    ref = OS.assemble(P, fmt="dense")
    for k in (1, 2, 5):
        a_ref = spla.lsqr(ref["M"], ref["h"], atol=0, btol=0, conlim=0, iter_lim=k)[0]
        with E.Solver.from_problem(P, precision=E.FP64) as s:
            s.assemble_problem(P)
            info = s.solve(preconditioner=E.PREC_NONE, max_iter=k, atol=0.0, btol=0.0,
                           check_every=1)
            a = s.coeffs()
        assert info.iterations == k
        assert np.linalg.norm(a - a_ref) <= 1e-10 * np.linalg.norm(a_ref)


@pytest.mark.parametrize("prec", [E.FP64, E.DF32])
@pytest.mark.parametrize("levels,K", [((1, 2, 4), 32), ((1, 2), 64), ((1, 2), 128)])
def test_block_jacobi_lsqr_iterates_match_preconditioned_lsqr(prec, levels, K):
    """With the block-Jacobi preconditioner the GPU runs LSQR on M P, P =
    diag_j R_j^{-1} with R_j^T R_j = G_jj + shift tr(G_jj)/K I and G_jj =
    M_j^T M_j (M_j: the K columns of subdomain j), and returns a = P y.  Its
    first iterates match SciPy's LSQR run on the same operator, built here in
    FP64 from the oracle's M.  This checks the preconditioner's set-up and its
    application inside the LSQR loop (both triangular products, the slice sums
    of M^T u, the update) value by value, for three block geometries.  The
    shift (1e-4) bounds cond(G_jj + shift) near 3e5, so that rounding-level
    differences in G_jj stay near 1e-10 in the iterates."""
    P = WL.poisson2d(levels=levels, features=K, n_side=40, n_boundary_side=40)
    ref = OS.assemble(P, fmt="dense")
    M, h = ref["M"], ref["h"]
    shift = 1e-4
    n = M.shape[1]
    Pm = np.zeros((n, n))
    for j in range(n // K):
        Mj = M[:, j * K:(j + 1) * K]
        G = Mj.T @ Mj
        L = np.linalg.cholesky(G + shift * np.trace(G) / K * np.eye(K))
        Pm[j * K:(j + 1) * K, j * K:(j + 1) * K] = np.linalg.inv(L.T)
    A = M @ Pm
    for k in (1, 2, 3):
        a_ref = Pm @ spla.lsqr(A, h, atol=0, btol=0, conlim=0, iter_lim=k)[0]
        with E.Solver.from_problem(P, precision=prec) as s:
            s.assemble_problem(P)
            info = s.solve(max_iter=k, atol=0.0, btol=0.0, check_every=1, shift=shift)
            a = s.coeffs()
        assert info.iterations == k
        err = np.linalg.norm(a - a_ref) / np.linalg.norm(a_ref)
        print(f"K={K} prec={prec} iterate {k}: relative difference {err:.2e}")
        assert err <= 1e-8


@pytest.mark.parametrize("prec", [E.FP64, E.FP32, E.DF32])
def test_block_cholesky_retries_with_a_larger_shift(prec):
    """Shift 0 on diagonal blocks of rank < K: the first factorisation meets a
    non-positive pivot, so the set-up starts again from a fresh copy of the
    block with the shift raised (1e-14 tr/K, then 100-fold), and the solve
    proceeds with finite coefficients.  NumPy's Cholesky confirms on the
    oracle's M that every block is singular at shift 0 and factorises at
    1e-14 tr/K."""
    K = 16
    P = WL.poisson1d(levels=(2, 4), features=K, n_interior=16)
    M = OS.assemble(P, fmt="dense")["M"]
    for j in range(M.shape[1] // K):
        Mj = M[:, j * K:(j + 1) * K]
        G = Mj.T @ Mj
        with pytest.raises(np.linalg.LinAlgError):
            np.linalg.cholesky(G)
        np.linalg.cholesky(G + 1e-14 * np.trace(G) / K * np.eye(K))
    with E.Solver.from_problem(P, precision=prec) as s:
        s.assemble_problem(P)
        info = s.solve(max_iter=20, atol=0.0, btol=0.0, shift=0.0, check_every=10)
        a = s.coeffs()
    assert info.iterations == 20
    assert info.precond_retries >= M.shape[1] // K   # every block retried at least once
    assert np.all(np.isfinite(a))


@pytest.mark.parametrize("prec", [E.FP32, E.FP64])
def test_block_cholesky_drops_the_oracles_dependent_columns(prec):
    """drop_tol on under-resolved subdomains (8 x 8 single-level, K = 32, about
    50 collocation points per support): the columns the GPU drops (their
    coefficients exactly 0, counted in precond_dropped) are those the oracle's
    Cholesky with dropping drops on the Gram blocks of the panels' own entries,
    except columns whose pivot ratio lies within a factor 2 of the threshold
    (the GPU's Gram rounds differently there)."""
    from oracle import krylov as KR
    K, drop, shift = 32, 1e-4, 1e-6
    P = WL.poisson2d(levels=(8,), features=K, n_side=20, n_boundary_side=20)
    with E.Solver.from_problem(P, precision=prec) as s:
        s.assemble_problem(P)
        M, _ = s.get_rows(np.arange(P.n_rows))
        info = s.solve(max_iter=5, atol=0.0, btol=0.0, shift=shift, drop_tol=drop,
                       check_every=5)
        a = s.coeffs()
    gpu_dropped = a == 0.0
    oracle_dropped = np.zeros_like(gpu_dropped)
    borderline = np.zeros_like(gpu_dropped)
    for j in range(M.shape[1] // K):
        Mj = M[:, j * K:(j + 1) * K]
        _, kept, ratio = KR.cholesky_dropping(Mj.T @ Mj, shift, drop)
        oracle_dropped[j * K:(j + 1) * K] = ~kept
        borderline[j * K:(j + 1) * K] = (ratio > 0.5 * drop) & (ratio < 2.0 * drop)
    print(f"dropped: gpu {gpu_dropped.sum()} (info {info.precond_dropped}), oracle "
          f"{oracle_dropped.sum()}, borderline {borderline.sum()} of {a.size}")
    assert info.precond_dropped == gpu_dropped.sum()
    assert oracle_dropped.sum() > a.size // 4          # the case is under-resolved
    assert np.all((gpu_dropped == oracle_dropped) | borderline)
    assert np.all(np.isfinite(a))


@pytest.mark.parametrize("prec", [E.FP32, E.DF32])
def test_device_stop_makes_iterations_independent_of_check_interval(prec):
    """With the pair tail the stopping tests run on the device after every
    iteration and the kernels of later iterations return at once: check
    intervals of 1, 7 and 10 give the same iteration count and bitwise the
    same coefficients (the count equals the first iteration whose test is met,
    which check_every = 1 finds directly)."""
    P = WL.poisson2d(levels=(1, 2, 4), features=32, n_side=50, n_boundary_side=50)
    out = []
    for ce in (1, 7, 10):
        with E.Solver.from_problem(P, precision=prec) as s:
            s.assemble_problem(P)
            info = s.solve(max_iter=3000, atol=0.0, btol=0.0, ntol=1e-2, shift=1e-6,
                           check_every=ce)
            out.append((info.iterations, s.coeffs()))
    print("iterations:", [o[0] for o in out])
    assert out[0][0] == out[1][0] == out[2][0] < 3000
    assert out[0][0] % 7 != 0 or out[0][0] % 10 != 0   # not both multiples of the intervals
    assert np.array_equal(out[0][1], out[1][1]) and np.array_equal(out[0][1], out[2][1])


_SOLVE_CASES = [
    ("poisson1d_J16_K64_N2000", WL.config_poisson1d),
    ("dho_L1-8_K24_N1000", lambda: WL.dho(levels=(1, 2, 4, 8), features=24, n_interior=1000)),
    ("poisson2d_L1-4_K64_N60", lambda: WL.poisson2d(levels=(1, 2, 4), features=64, n_side=60,
                                                    n_boundary_side=60)),
]


_QR_CASES = _SOLVE_CASES + [
    ("dho_L1-64_K96_N20000", WL.config_dho_ml),
    ("helmholtz_L_w8_J16_K16", WL.helmholtz_lshape),      # §4.4, L-shaped domain
    ("laplace_n4_J16_K16", WL.laplace_multiscale),        # §4.3, hard-constraint ansatz
]


@pytest.mark.parametrize("name,make,prec", [(n, m, p) for n, m in _QR_CASES
                                            for p in (E.FP64, E.DF32)])
def test_solution_matches_oracle_qr_minimiser(name, make, prec):
    """The GPU's column-pivoted QR on the assembled system reaches the
    oracle's QR error (1.01x its largest value over row orders, plus the
    spread of those values: on the full DHO the minimiser's error is FP64
    rounding, 1.7e-14 to 2.4e-14 over three row orders, so 1% of it is below
    what reordering alone changes; elsewhere the spread is about 1e-12 of the
    error), with a numerical rank within the oracle's range over those orders
    (+-2: a pivot near the rank cut may fall either side of it)."""
    g = _golden(name)
    if "qr" not in g or "rel_l2_max_over_orders" not in g["qr"]:
        pytest.skip(f"{name}: no QR entry over row orders in oracle_errors.json")
    q = g["qr"]
    P = make()
    with E.Solver.from_problem(P, precision=prec) as s:
        s.assemble_problem(P)
        info = s.solve(method=E.SOLVE_QR)
        uh = s.eval(P.test_points)
        err = s.error_norms(uh, P.exact(P.test_points))
    ranks = [q["rank"]] + [o["rank"] for o in q["orders"]]
    print(f"{name} prec={prec}: gpu QR rel L2 {err['rel_l2']:.4e} rank {info.rank} "
          f"({info.solve_ms:.1f} ms, residual {info.residual_norm:.4e}); oracle QR "
          f"{q['rel_l2']:.4e}, max over orders {q['rel_l2_max_over_orders']:.4e}, "
          f"ranks {ranks}, residual {q['residual']:.4e}")
    errs = [q["rel_l2"]] + [o["rel_l2"] for o in q["orders"]]
    assert err["rel_l2"] <= 1.01 * q["rel_l2_max_over_orders"] + (max(errs) - min(errs))
    assert min(ranks) - 2 <= info.rank <= max(ranks) + 2
    assert info.residual_norm <= 1.01 * max([q["residual"]] + [o["residual"] for o in q["orders"]])


@pytest.mark.parametrize("prec", [E.FP32])
def test_full_size_2d_multilevel_solve_meets_paper_protocol(prec):
    """The 2-D multilevel Poisson workload at full size (161,600 rows, 43,648
    columns; its dense form, 56 GB, is beyond the oracle's memory, so its bar
    is the oracle's paper-protocol error, LSQR-15000 from the CSR system): the
    GPU's LSQR on FP32 panels stopped by its own normal-residual test (1e-4).
    (Its FP32-pair panels are outside the pair pass's limits: 17 covering
    panels x K = 128 per cell.)"""
    g = _golden("poisson2d_L1-16_K128_N400")
    P = WL.config_poisson2d_ml()
    with E.Solver.from_problem(P, precision=prec) as s:
        s.assemble_problem(P)
        info = s.solve(max_iter=5000, atol=0.0, btol=0.0, ntol=1e-4, shift=1e-6,
                       check_every=10)
        err = s.error_norms(s.eval(P.test_points), P.exact(P.test_points))["rel_l2"]
    print(f"2-D multilevel, full size, prec {prec}: rel L2 {err:.3e} ({info.iterations} its); "
          f"oracle LSQR-15000 {g['lsqr']['rel_l2']:.3e}")
    assert info.status == E.OK
    assert err <= 1.01 * g["lsqr"]["rel_l2"]


def test_qr_full_rank_coefficients_match_oracle():
    """A small full-rank system (kappa ~ 1e4): the least-squares solution is
    unique, so the GPU QR's coefficients equal the oracle QR's."""
    from oracle import lstsq as OL
    P = WL.poisson1d(levels=(4,), features=4, n_interior=200, lam=100.0)
    ref = OS.assemble(P, fmt="dense")
    a_ref, rank = OL.lstsq_qr(ref["M"], ref["h"])
    assert rank == P.n_columns
    with E.Solver.from_problem(P, precision=E.FP64) as s:
        s.assemble_problem(P)
        info = s.solve(method=E.SOLVE_QR)
        a = s.coeffs()
    assert info.rank == rank and info.iterations == rank
    assert np.linalg.norm(a - a_ref) <= 1e-11 * np.linalg.norm(a_ref)
    assert info.residual_norm == pytest.approx(np.linalg.norm(ref["M"] @ a_ref - ref["h"]),
                                               rel=1e-10)


def test_qr_rank_deficient_fit_matches_oracle():
    """Rank deficient (overlapping subdomains, 16 features each): the fitted
    values M a and the residual are unique and match the oracle's."""
    from oracle import lstsq as OL
    P = WL.dho(levels=(1, 2, 4), features=16, n_interior=300, omega0=10.0)
    ref = OS.assemble(P, fmt="dense")
    M, h = ref["M"], ref["h"]
    a_ref, rank = OL.lstsq_qr(M, h)
    with E.Solver.from_problem(P, precision=E.FP64) as s:
        s.assemble_problem(P)
        info = s.solve(method=E.SOLVE_QR)
        a = s.coeffs()
    print(f"rank gpu {info.rank} oracle {rank} of {M.shape[1]}")
    assert abs(info.rank - rank) <= 1
    fit, fit_ref = M @ a, M @ a_ref
    assert np.linalg.norm(fit - fit_ref) <= 1e-9 * np.linalg.norm(h)
    assert np.linalg.norm(fit - h) == pytest.approx(np.linalg.norm(fit_ref - h), rel=1e-6)


def test_qr_rejects_a_dense_matrix_beyond_device_memory():
    """The 2-D multilevel Poisson workload at 400^2 (161,600 x 43,649 dense,
    56 GB) fits a GB300; a 1024^2 grid with 4096 subdomains of 32 features
    would not (1.1 TB): UNSUPPORTED before anything is allocated."""
    P = WL.poisson2d(levels=(64,), features=32, n_side=1024, n_boundary_side=8)
    with E.Solver.from_problem(P, precision=E.FP32) as s:
        s.assemble_problem(P)
        with pytest.raises(E.ElmfbError) as ei:
            s.solve(method=E.SOLVE_QR)
        assert ei.value.code == E.ERR_UNSUPPORTED


@pytest.mark.parametrize("name,make,prec", [(n, m, p) for n, m in _SOLVE_CASES + [
    ("helmholtz_L_w8_J16_K16", WL.helmholtz_lshape),
    ("laplace_n4_J16_K16", WL.laplace_multiscale)] for p in (E.FP64, E.DF32)])
def test_block_jacobi_lsqr_meets_paper_protocol_error(name, make, prec):
    g = _golden(name)
    P = make()
    with E.Solver.from_problem(P, precision=prec) as s:
        s.assemble_problem(P)
        info = s.solve(max_iter=15000, atol=1e-14, btol=1e-14, shift=1e-12)
        uh = s.eval(P.test_points)
        err = s.error_norms(uh, P.exact(P.test_points))
    print(f"{name}: gpu rel L2 {err['rel_l2']:.3e} ({info.iterations} its, "
          f"{info.solve_ms:.1f} ms); oracle LSQR-15000 {g['lsqr']['rel_l2']:.3e}; "
          f"oracle QR {g.get('qr', {}).get('rel_l2', float('nan')):.3e}")
    # LSQR converges to the least-squares minimiser; where the paper's
    # unconverged 15000th iterate happens to lie closer to u than the minimiser
    # (Helmholtz: 2.73e-2 against 2.78e-2), the minimiser's own error is the bar
    qr = g.get("qr", {}).get("rel_l2_max_over_orders", 0.0)
    assert err["rel_l2"] <= 1.01 * max(g["lsqr"]["rel_l2"], qr)


@pytest.mark.parametrize("make", [
    lambda: WL.helmholtz_lshape(levels=(1, 8), features=12, n_grid=30, n_long=30, n_short=15),
    lambda: WL.laplace_multiscale(omegas=(3, 5), levels=(1, 4), features=12, n_grid=20)])
def test_eval_matches_oracle_u_hat_with_holes_and_ansatz(make):
    """u_hat of the L-shaped domain (discarded subdomains) and of the
    hard-constraint ansatz (u~ = A u_hat) at the test points, at the box
    boundary (where the ansatz vanishes) and at random interior points."""
    from oracle import decomposition as OD
    P = make()
    a = np.random.default_rng(3).standard_normal(OD.n_columns(P))
    X = np.concatenate([P.test_points, WL.square_boundary_midpoints(5)])
    if P.holes:
        X = X[~((X[:, 0] > 0.5) & (X[:, 1] > 0.5))]
    with E.Solver.from_problem(P, precision=E.FP64) as s:
        s.set_coeffs(a)
        uh = s.eval(X)
    ref = OE.u_hat(P, a, X)
    assert np.allclose(uh, ref, rtol=1e-12, atol=1e-12 * np.abs(ref).max())
    if P.ansatz_omega:
        nb = WL.square_boundary_midpoints(5).shape[0]
        assert np.all(uh[-nb:] == 0.0)


def test_eval_matches_oracle_u_hat():
    P = WL.poisson2d(levels=(1, 2, 4), features=24, n_side=20, n_boundary_side=10, delta=2.9)
    a = np.random.default_rng(1).standard_normal(P.n_columns)
    X = np.concatenate([P.test_points, np.array([[0.0, 0.0], [1.0, 1.0], [0.5, 0.25]])])
    with E.Solver.from_problem(P, precision=E.FP64) as s:
        s.set_coeffs(a)
        uh = s.eval(X)
    ref = OE.u_hat(P, a, X)
    assert np.allclose(uh, ref, rtol=1e-12, atol=1e-12 * np.abs(ref).max())


def test_full_size_large_2d_solution_evaluates_as_the_oracle_model():
    """The large 2-D multilevel workload (4.2M rows, 349,504 columns: beyond
    any oracle solve) solved as the bench does; the oracle evaluates the model
    with the GPU's coefficients at 256 sampled test points, one by one, and
    the GPU's u_hat agrees to FP64 rounding of the terms (the windows of a
    level sum to 1 and |tanh| <= 1, so a point's terms add up in magnitude to
    at most max_j ||a_j||_1).  The GPU's error norms against the closed form
    equal the oracle's on the same u_hat."""
    P = WL.config_poisson2d_large()
    rng = np.random.default_rng(5)
    X = P.test_points[rng.choice(P.test_points.shape[0], 256, replace=False)]
    with E.Solver.from_problem(P, precision=E.FP32) as s:
        s.assemble_problem(P)
        info = s.solve(max_iter=5000, atol=0.0, btol=0.0, ntol=1e-4, shift=1e-6, check_every=10)
        a = s.coeffs()
        uh = s.eval(X)
        u = P.exact(X)
        norms = s.error_norms(uh, u)
    ref = OE.u_hat(P, a, X)
    scale = np.abs(a).reshape(-1, P.features).sum(axis=1).max()
    diff = np.abs(uh - ref).max()
    print(f"{info.iterations} its; sampled rel L2 {norms['rel_l2']:.3e}; |gpu - oracle| {diff:.3e}"
          f" (term scale {scale:.3e})")
    assert diff <= 1e-13 * scale + 1e-12 * np.abs(ref).max()
    assert norms["rel_l2"] == pytest.approx(OE.rel_l2(uh, u), rel=1e-12)
    assert norms["e_l1"] == pytest.approx(OE.e_l1(uh, u), rel=1e-12)


def test_error_norms_match_oracle():
    rng = np.random.default_rng(2)
    u = rng.standard_normal(10007)
    uh = u + 1e-3 * rng.standard_normal(u.size)
    P = WL.poisson1d(levels=(2,), features=4, n_interior=10)
    with E.Solver.from_problem(P) as s:
        out = s.error_norms(uh, u)
    assert out["rel_l2"] == pytest.approx(OE.rel_l2(uh, u), rel=1e-12)
    assert out["e_l1"] == pytest.approx(OE.e_l1(uh, u), rel=1e-12)
    assert out["max_abs"] == pytest.approx(np.abs(uh - u).max(), rel=1e-15)


def test_iteration_cap_reports_not_converged_with_valid_coefficients():
    P = WL.config_poisson1d()
    with E.Solver.from_problem(P, precision=E.FP64) as s:
        s.assemble_problem(P)
        info = s.solve(max_iter=7, atol=1e-30, btol=1e-30, check_every=3)
        assert info.status == E.ERR_NOT_CONVERGED and info.iterations == 7
        assert np.all(np.isfinite(s.coeffs()))


def test_solve_before_assemble_is_state_error():
    P = WL.poisson1d(levels=(2,), features=4, n_interior=10)
    with E.Solver.from_problem(P) as s:
        with pytest.raises(E.ElmfbError) as ei:
            s.solve()
        assert ei.value.code == E.ERR_STATE


def test_warm_start_continues_from_coefficients():
    P = WL.dho(levels=(1, 2, 4), features=16, n_interior=400, omega0=15.0)
    with E.Solver.from_problem(P, precision=E.FP64) as s:
        s.assemble_problem(P)
        s.solve(max_iter=40, atol=0, btol=0)
        r40 = _residual(s, P)
        s.solve(max_iter=40, atol=0, btol=0, warm_start=1)
        r80 = _residual(s, P)
    assert r80 < r40


def _residual(s, P):
    ref = OS.assemble(P, fmt="dense")
    return float(np.linalg.norm(ref["M"] @ s.coeffs() - ref["h"]))


def test_fp32_panels_solution_vs_paper_protocol():
    """FP32 panels on the 2-D multilevel Poisson case beat the paper's protocol.

    (On the damped oscillator FP32 storage of M itself is the limit: the exact
    least-squares solution of the FP32-rounded matrix is already less accurate
    than the paper protocol -- see tests/test_oracle_precision.py -- so that
    workload runs with FP64 panels.)"""
    name = "poisson2d_L1-4_K64_N60"
    g = _golden(name)
    P = WL.poisson2d(levels=(1, 2, 4), features=64, n_side=60, n_boundary_side=60)
    errs = {}
    for prec in (E.FP64, E.FP32):
        with E.Solver.from_problem(P, precision=prec) as s:
            s.assemble_problem(P)
            s.solve(max_iter=5000, atol=1e-12, btol=1e-12, shift=1e-10)
            errs[prec] = s.error_norms(s.eval(P.test_points), P.exact(P.test_points))["rel_l2"]
    print("fp64 / fp32 rel L2:", errs, "oracle LSQR-15000:", g["lsqr"]["rel_l2"])
    assert errs[E.FP64] <= 1.01 * g["lsqr"]["rel_l2"]
    assert errs[E.FP32] <= 1.01 * g["lsqr"]["rel_l2"]


@pytest.mark.parametrize("prec", [E.FP32, E.FP64])
@pytest.mark.parametrize("variant", ["pipe8", "pipe4", "registers"])
def test_both_fused_pass_variants_meet_paper_protocol_error(prec, variant, monkeypatch):
    """The fused LSQR pass has a shared-memory pipelined form (bulk copies of
    8-row chunks, or 4-row chunks when three 8-row stages do not fit; FP32
    sums of the per-panel dots for FP32 panels) and a register-load form (the
    fallback when the ring does not fit); each meets the solution bar on its
    own."""
    g = _golden("poisson2d_L1-4_K64_N60")
    P = WL.poisson2d(levels=(1, 2, 4), features=64, n_side=60, n_boundary_side=60)
    monkeypatch.setenv("ELMFB_FUSED_REGISTERS", "1" if variant == "registers" else "0")
    if variant == "pipe4":
        monkeypatch.setenv("ELMFB_FUSED_ROWS", "4")
    with E.Solver.from_problem(P, precision=prec) as s:
        s.assemble_problem(P)
        info = s.solve(max_iter=4000, atol=1e-14, btol=1e-14, shift=1e-12)
        err = s.error_norms(s.eval(P.test_points), P.exact(P.test_points))["rel_l2"]
    print(f"{variant} prec={prec}: rel L2 {err:.3e} ({info.iterations} its); "
          f"oracle LSQR-15000 {g['lsqr']['rel_l2']:.3e}")
    assert err <= 1.01 * g["lsqr"]["rel_l2"]


def test_df32_solve_needs_features_multiple_of_four():
    """The DF32 solvers need K a multiple of 4 (16-byte vector reads of FP32
    pairs, 4x4 Gram tiles): K = 33 is rejected before any solver kernel runs;
    the assembly itself works for any K."""
    P = WL.poisson2d(levels=(1, 3), features=33, n_side=30, n_boundary_side=10)
    with E.Solver.from_problem(P, precision=E.DF32) as s:
        s.assemble_problem(P)
        with pytest.raises(E.ElmfbError) as ei:
            s.solve(max_iter=10)
        assert ei.value.code == E.ERR_UNSUPPORTED


def test_profiling_stride_times_every_nth_launch():
    """elmfb_set_profiling_stride: with profiling restricted to the fused pass
    and stride 4, the handle times launches 0, 4, 8, ... of that kernel only
    (the bench times its roofline kernel this way); stride 0 is rejected."""
    P = WL.poisson2d(levels=(1, 2), features=32, n_side=30, n_boundary_side=30)
    with E.Solver.from_problem(P, precision=E.FP32) as s:
        s.assemble_problem(P)
        s.set_profiling_only("fused_Mt_MTu")
        with pytest.raises(E.ElmfbError) as ei:
            s.set_profiling_stride(0)
        assert ei.value.code == E.ERR_INVALID_ARG
        s.set_profiling_stride(4)
        info = s.solve(max_iter=13, atol=0.0, btol=0.0, check_every=13)
        stats = s.kernel_stats()
    # one fused pass for the start plus one per iteration
    passes = 1 + info.iterations
    ms, timed, _ = stats["fused_Mt_MTu"]
    assert timed == (passes + 3) // 4
    assert ms > 0.0
    assert set(stats) == {"fused_Mt_MTu"}


@pytest.mark.parametrize("n", [20, 200, 2030, 2046, 2078, 4200])
def test_qr_over_row_counts(n):
    """The QR update holds a column in registers once at most 2048 rows are left
    and reads it twice before that: systems of fewer rows than columns (20), well
    below, at and just past the limit (cells are padded to 16 rows), and far past
    it, against the oracle's QR: the rank to one (a pivot may sit at the cut) and
    the error to half as much again (two orders of the same rows differ by less
    in the golden workloads)."""
    from oracle import lstsq as OL
    from oracle import system as OS
    P = WL.poisson1d(levels=(1, 4), features=12, n_interior=n, lam=1e4)
    ref = OS.assemble(P, fmt="dense")
    a_o, rank = OL.lstsq_qr(ref["M"], ref["h"])
    with E.Solver.from_problem(P, precision=E.FP64) as s:
        s.assemble_problem(P)
        info = s.solve(method=E.SOLVE_QR)
        a = s.coeffs()
    assert abs(info.rank - rank) <= 1
    r, r_o = (np.linalg.norm(ref["M"] @ v - ref["h"]) for v in (a, a_o))
    h = np.linalg.norm(ref["h"])
    assert r <= 1.5 * r_o + 1e-9 * h


@pytest.mark.parametrize("K", [8, 24, 32, 56, 72, 104, 128])
def test_block_jacobi_factors_over_feature_counts(K):
    """Preconditioned LSQR on FP32 panels at feature counts multiple of 8 (the
    packed 4 x 8 tiles of the diagonal Gram blocks: one tile column, ragged last
    warps, the largest): with a shift of 1e-2 the first iterate depends on the
    blocks only to FP32 accuracy times the shift's inverse, 100 x 2^-24 x (a few
    roundings) < 1e-4 of the one that SciPy gives with the oracle's FP64 blocks."""
    from oracle import system as OS
    P = WL.poisson2d(levels=(1, 2), features=K, n_side=37, n_boundary_side=12)
    ref = OS.assemble(P, fmt="dense")
    M, h, ns = ref["M"], ref["h"], P.n_subdomains
    X = np.zeros((ns * K, ns * K))
    for j in range(ns):
        b = slice(j * K, (j + 1) * K)
        G = M[:, b].T @ M[:, b]
        L = np.linalg.cholesky(G + 1e-2 * np.trace(G) / K * np.eye(K))
        X[b, b] = np.linalg.inv(L).T
    a_ref = X @ spla.lsqr(M @ X, h, atol=0, btol=0, conlim=0, iter_lim=1)[0]
    with E.Solver.from_problem(P, precision=E.FP32) as s:
        s.assemble_problem(P)
        s.solve(max_iter=1, atol=0.0, btol=0.0, shift=1e-2, check_every=1)
        a = s.coeffs()
    assert np.linalg.norm(a - a_ref) <= 1e-4 * np.linalg.norm(a_ref)


def test_autotuned_units_do_not_depend_on_other_systems():
    """Two FP64 systems of one precision, K, covering panels and log2 of the rows:
    17 cells (few units: about one per SM, 8 to 32 rows) and 81 cells of 48 rows
    (every candidate, 256 rows and more, makes a cell one unit).  Tuned after the
    first, the second solves bit for bit as untuned."""
    P = [WL.poisson1d(levels=(n,), features=56, n_interior=r) for n, r in ((16, 2000), (80, 3300))]
    out = []
    for tune in (0, 1):
        for p in P[1 - tune:]:
            with E.Solver.from_problem(p, precision=E.FP64) as s:
                s.assemble_problem(p)
                s.solve(preconditioner=E.PREC_NONE, max_iter=12, atol=0.0, btol=0.0, autotune=tune)
                out.append(s.coeffs())
    assert np.array_equal(out[0], out[2])
    tuned = [e for e in E.tuning_table() if e["precision"] == E.FP64 and e["features"] == 56]
    assert len({e["rows_log2"] for e in tuned}) == 1 and len(tuned) == 2
