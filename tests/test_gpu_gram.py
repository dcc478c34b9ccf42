"""GPU parity of the tensor-core Gram blocks G_ij = M_i^T M_j.

Two references from the oracle's FP64 matrix M (never from the GPU):
* G_bf = bf16(M)^T bf16(M) in FP64 (M rounded to BF16 by torch): the
  tensor cores multiply these BF16 values and accumulate in FP32; the GPU
  rounds its own FP32 entries, so an entry next to a rounding boundary can
  land one BF16 ulp away from the oracle's rounding.  Bound used:
  |G - G_bf| <= 2^-9 |M|^T|M|, a quarter of the worst-case rounding bound
  below (an operand layout error would show as O(1));
* G = M^T M in FP64: |G_gpu - G| <= (2 u_bf16 + u_bf16^2) |M|^T|M| + FP32
  accumulation, u_bf16 = 2^-8 (the worst-case rounding bound).
"""
import numpy as np
import pytest

import paper_2409_01949_gb300 as E
import workloads as WL
from oracle import system as OS

pytestmark = pytest.mark.gpu

CASES = {
    "poisson2d_L1-4_K64": lambda: WL.poisson2d(levels=(1, 2, 4), features=64, n_side=40,
                                               n_boundary_side=40),
    "poisson2d_L1-2_K128": lambda: WL.poisson2d(levels=(1, 2), features=128, n_side=24,
                                                n_boundary_side=12),
    "dho_L1-8_K24": lambda: WL.dho(levels=(1, 2, 4, 8), features=24, n_interior=700),
    "poisson2d_delta2.9_K40": lambda: WL.poisson2d(levels=(2, 3), features=40, n_side=30,
                                                   n_boundary_side=10, delta=2.9),
}


def _bf16(A):
    torch = pytest.importorskip("torch")
    return torch.from_numpy(A.astype(np.float32)).bfloat16().double().numpy()


@pytest.mark.parametrize("name", list(CASES))
def test_gram_blocks_match_oracle(name):
    P = CASES[name]()
    K = P.features
    ref = OS.assemble(P, fmt="dense")
    M = ref["M"]
    Mb = _bf16(M)
    A = np.abs(M)
    nsub = P.n_subdomains
    # structural pairs from the oracle: blocks of M^T M with a shared row
    nzb = (np.abs(M).reshape(M.shape[0], nsub, K).max(axis=2) > 0)
    share = (nzb.T.astype(np.int64) @ nzb.astype(np.int64)) > 0
    pairs = [(i, j) for i in range(nsub) for j in range(i, nsub) if share[i, j]]
    with E.Solver.from_problem(P, precision=E.MIXED) as s:
        s.assemble_problem(P)
        s.compute_gram()
        sz = s.sizes()
        got = s.gram_blocks(pairs)
    assert sz.n_gram_pairs >= len(pairs)
    worst_bf, worst_ex = 0.0, 0.0
    for q, (i, j) in enumerate(pairs):
        bi, bj = slice(i * K, (i + 1) * K), slice(j * K, (j + 1) * K)
        Gabs = A[:, bi].T @ A[:, bj]
        Gbf = Mb[:, bi].T @ Mb[:, bj]
        Gex = M[:, bi].T @ M[:, bj]
        sc = np.maximum(Gabs, 1e-300)
        worst_bf = max(worst_bf, float((np.abs(got[q] - Gbf) / sc).max()))
        worst_ex = max(worst_ex, float((np.abs(got[q] - Gex) / sc).max()))
    print(f"{name}: {len(pairs)} pairs, max |G-G_bf16|/|M|^T|M| = {worst_bf:.2e}, "
          f"max |G-G|/|M|^T|M| = {worst_ex:.2e}")
    assert worst_bf <= 2.0 ** -9
    assert worst_ex <= 2 * 2.0 ** -8 + 2.0 ** -16 + 1e-4


def test_gram_unsupported_outside_mixed_precision():
    P = WL.poisson1d(levels=(2,), features=8, n_interior=20)
    with E.Solver.from_problem(P, precision=E.FP32) as s:
        s.assemble_problem(P)
        with pytest.raises(E.ElmfbError) as ei:
            s.compute_gram()
        assert ei.value.code == E.ERR_UNSUPPORTED


# K below one MMA's granularity, ragged against 4, 8 and 16, and the largest; the
# level-1 subdomain's rows span several tasks, a (1,)-level problem is one pair
@pytest.mark.parametrize("levels,K,side", [((1,), 1, 9), ((1, 3), 17, 30), ((1, 2, 4), 100, 50),
                                           ((5,), 36, 41), ((1, 2), 128, 33)])
def test_gram_blocks_of_cut_pairs(levels, K, side):
    """Every block, asked for in either order and into host or device memory,
    with a pair that shares no rows, against BF16-rounded products in FP64
    (bound of the module's first reference)."""
    torch = pytest.importorskip("torch")
    P = WL.poisson2d(levels=levels, features=K, n_side=side, n_boundary_side=side)
    M = OS.assemble(P, fmt="dense")["M"]
    Mb, A, nsub = _bf16(M), np.abs(M), P.n_subdomains
    pairs = [(i, j) if (i + j) % 2 else (j, i) for i in range(nsub) for j in range(i, nsub)]
    with E.Solver.from_problem(P, precision=E.MIXED) as s:
        s.assemble_problem(P)
        s.compute_gram()
        got = s.gram_blocks(pairs)
        p = np.array(pairs, dtype=np.int32)
        dev = torch.empty((len(p), K, K), dtype=torch.float64, device="cuda")
        assert E.lib().elmfb_get_gram(s.h, len(p), p.ctypes.data, dev.data_ptr()) == E.OK
        s.compute_gram()   # the plan is kept, the blocks are the same
        again = s.gram_blocks(pairs)
    assert np.array_equal(dev.cpu().numpy(), got) and np.array_equal(again, got)
    for q, (i, j) in enumerate(pairs):
        bi, bj = slice(i * K, (i + 1) * K), slice(j * K, (j + 1) * K)
        assert np.all(np.abs(got[q] - Mb[:, bi].T @ Mb[:, bj]) <=
                      2.0 ** -9 * (A[:, bi].T @ A[:, bj]))


@pytest.mark.parametrize("make", [
    lambda: WL.poisson1d(levels=(1, 3, 5), features=4, n_interior=90),
    lambda: WL.poisson1d(levels=(7,), features=4, n_interior=5, delta=2.9),       # empty cells
    lambda: WL.poisson2d(levels=(1, 2, 4, 8), features=4, n_side=40),
    lambda: WL.poisson2d(levels=(3, 5), features=4, n_side=24, delta=1.4),
    lambda: WL.poisson2d(levels=(2, 6), features=4, n_side=5, delta=2.9),         # empty cells
    lambda: WL.helmholtz_lshape(levels=(1, 8), features=4, n_grid=20),            # discarded subdomains
    lambda: WL.laplace_multiscale(levels=(1, 4, 6), features=4, n_grid=30, placement="endpoint"),
])
def test_pair_count_before_and_after_the_gram_blocks(make):
    """sizes() counts the pairs of subdomains that share a cell with points
    without forming them; the blocks' own list has the same number."""
    P = make()
    with E.Solver.from_problem(P, precision=E.MIXED) as s:
        s.assemble_problem(P)
        n = s.sizes().n_gram_pairs
        s.compute_gram()
        assert s.sizes().n_gram_pairs == n


def _scattered(n, box, seed):
    r = np.random.default_rng(seed)
    lo, hi = np.array(box[0]), np.array(box[1])
    return lo + (hi - lo) * r.random((n, 2))


@pytest.mark.parametrize("K,n", [(32, 40000), (128, 40000)])
def test_gram_block_depends_on_its_own_rows_only(K, n):
    """A pair's block is one accumulation over its rows: the blocks of the
    subdomains left of x = 0.5 have the same bits whether the other half of the
    domain holds a few points or most of them.  (The second system has four
    times the interior points, so its rows are scaled by exactly 1/2.)

    They also agree with the FP64 products of the rounded operands -- BF16 of
    the panels' own FP32 entries -- to FP32 accumulation over steps of 16 rows,
    each step truncated at 2^-23 of the accumulated magnitude in each of its
    partial sums (2^-22 a step): a lost row of a pair's thousands would
    show."""
    left = _scattered(n, ((0.0, 0.0), (0.45, 1.0)), 1)
    few = _scattered(n // 8, ((0.75, 0.0), (1.0, 1.0)), 2)
    many = _scattered(4 * (n + n // 8) - n, ((0.75, 0.0), (1.0, 1.0)), 3)
    # single level, 4 x 4 subdomains of half-width 1/4: those of columns 0 and 1
    # end at x = 0.625
    pairs = [(0, 0), (0, 1), (1, 5), (4, 5), (9, 9), (8, 13)]
    out, T = [], None
    for right in (few, many):
        x = np.concatenate([left, right])
        with E.Solver(2, (0.0, 0.0), (1.0, 1.0), (4,), 2.0, K, precision=E.MIXED) as s:
            s.assemble([dict(points=x, rhs=np.zeros(len(x)), c2=(-1.0, -1.0))])
            s.compute_gram()
            out.append(s.gram_blocks(pairs))
            if T is None:
                T = s.get_rows(np.arange(n))[0]
    assert np.array_equal(out[0], 4.0 * out[1])
    B = _bf16(T)
    for q, (i, j) in enumerate(pairs):
        bi, bj = B[:, i * K:(i + 1) * K], B[:, j * K:(j + 1) * K]
        # rows of cells that the supports share, padded to 16 a cell (16 cells at most)
        steps = np.count_nonzero(np.abs(bi).any(1) & np.abs(bj).any(1)) / 16 + 16
        mag = np.abs(bi).T @ np.abs(bj)
        assert np.all(np.abs(out[0][q] - bi.T @ bj) <= steps * 2.0 ** -22 * mag)


def test_blocks_to_the_host_take_little_device_memory():
    """600 MB of blocks asked for into host memory pass through a bounded buffer
    (32 MB; the library's pool keeps what it has taken, so the free memory shows it)."""
    torch = pytest.importorskip("torch")
    P = WL.poisson2d(levels=(2,), features=128, n_side=12, n_boundary_side=4)
    pairs = [(q % 4, (q // 4) % 4) for q in range(4601)]
    with E.Solver.from_problem(P, precision=E.MIXED) as s:
        s.assemble_problem(P)
        s.compute_gram()
        few = s.gram_blocks(pairs[:16])
        E.trim_memory()
        before = torch.cuda.mem_get_info()[0]
        got = s.gram_blocks(pairs)
        taken = before - torch.cuda.mem_get_info()[0]
    assert taken <= 128 << 20
    for q in range(0, 4601, 16):
        assert np.array_equal(got[q:q + 16], few[:4601 - q])


def test_blocks_in_place_come_after_pending_work_on_the_buffer():
    """A handle on a stream of its own writes blocks into a device buffer that the
    default stream is still to fill: the blocks are what remains, as after a copy."""
    torch = pytest.importorskip("torch")
    P = WL.poisson2d(levels=(2,), features=64, n_side=12, n_boundary_side=4)
    p = np.array([(0, 0), (0, 3), (1, 2)], dtype=np.int32)
    side = torch.cuda.Stream()
    with E.Solver.from_problem(P, precision=E.MIXED, stream=side.cuda_stream) as s:
        s.assemble_problem(P)
        s.compute_gram()
        want = s.gram_blocks(p)
        out = torch.zeros((3, 64, 64), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        torch.cuda._sleep(100_000_000)   # some 50 ms
        out.fill_(7.0)
        assert E.lib().elmfb_get_gram(s.h, 3, p.ctypes.data, out.data_ptr()) == E.OK
        torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy(), want)
