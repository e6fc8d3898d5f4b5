"""The blocked dense LDL^T of S at the edges of its panels and tiles, by its
backward error.  Without pivoting the computed factors of a matrix of order n
satisfy |L D L^T - S| <= c n u |L| |D| |L|^T entry by entry (u the unit
roundoff, c a small constant: 4 covers the reciprocal and the two roundings of
a product with it), whatever the order of the operations."""
import numpy as np
import pytest

from gen import GridSpec, make_problem

pytestmark = pytest.mark.gpu


def _torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def dense_c(n, seed):
    """A tiny system whose S is C itself (B = 0): symmetric, quasidefinite
    (half its pivots negative) and with entries over a few decades."""
    from dataclasses import replace

    p = make_problem(GridSpec(5, 6, 2, 1, 3, 1e-1, 1e1, 7, "tiny"), zero_b=True)
    rng = np.random.default_rng(seed)
    s = np.where(rng.random(n) < 0.5, -1.0, 1.0)
    m = rng.standard_normal((n, n)) * 10.0 ** rng.uniform(-1, 0, (n, 1))
    m = (m + m.T) / 2
    m[np.ix_(s > 0, s > 0)] /= 2
    m[np.ix_(s < 0, s < 0)] /= 2
    m[np.diag_indices(n)] = s * (1.0 + np.abs(m).sum(1) * 0.6)
    nC = n
    b_blockptr = np.arange(p.N + 1, dtype=np.int32)
    b_row = np.full(p.N, p.nA - 1, dtype=np.int32)
    b_col = (np.arange(p.N) % nC).astype(np.int32)
    rhs = rng.standard_normal(p.N * p.nA + nC)
    return replace(p, nC=nC, c_kind=1, c_vals=m.reshape(-1).copy(), b_blockptr=b_blockptr, b_row=b_row, b_col=b_col,
                   b_vals=np.zeros(p.N), rhs=rhs), m


@pytest.mark.parametrize("prec", ["fp64", "tf32"])
@pytest.mark.parametrize("n", [1, 15, 16, 17, 31, 32, 33, 48, 63, 64, 65, 100, 129, 300])
def test_factor_of_s_backward_error(n, prec):
    torch = _torch()
    from paper_1907_05420_gb300 import binding as B

    if prec == "tf32" and n > 64:
        pytest.skip("the trailing updates of TF32 round their operands")
    p, m = dense_c(n, 100 + n)
    up = lambda v: torch.from_numpy(np.ascontiguousarray(v)).to("cuda:0")  # noqa: E731
    h = B.kkt_analyze(p, B.kkt_default_options(prec))
    try:
        B.kkt_factor(h, up(p.a_vals), up(p.b_vals), up(p.c_vals))
        out = torch.empty(n * n, dtype=torch.float64, device="cuda:0")
        B.kkt_schur_factor_copy(h, out)
        info = B.kkt_get_info(h)
        f = out.cpu().numpy().reshape(n, n).T.astype(np.longdouble)
    finally:
        B.kkt_destroy(h)
    d = np.diag(f).copy()
    lo = np.tril(f, -1) + np.eye(n)
    s = m.astype(np.float32 if prec == "tf32" else np.float64).astype(np.longdouble)
    u = 2.0 ** -24 if prec == "tf32" else 2.0 ** -53
    diff = np.abs(np.tril(lo * d @ lo.T - s))
    assert np.all(diff <= 4 * (n + 2) * u * (np.abs(lo) * np.abs(d) @ np.abs(lo).T))
    neg = int((np.linalg.eigvalsh(m) < 0).sum())
    assert info["n_neg"] == p.N * (p.nA - p.nP) + neg and info["n_zero"] == 0


@pytest.mark.parametrize("prec,s", [("fp64", 0), ("fp64", 1), ("f64emu", 0), ("tf32", 0)])
@pytest.mark.parametrize("n", [1, 63, 64, 65, 128, 129, 200, 577])
def test_solve_with_s(n, prec, s):
    """The chain of 64-row blocks of the triangular solves: with B = 0 the
    coupling part of the solution is S^{-1} r_g alone.  The FP64-accurate
    factors meet the backward error of the whole system (||K|| includes |S|)
    without refinement: 4 (n + 2) u with the growth |L||D||L|^T <= 4 |S| of
    these diagonally dominant matrices; the FP32 factor with it."""
    torch = _torch()
    import oracle
    from paper_1907_05420_gb300 import binding as B

    p, m = dense_c(n, 300 + n)
    up = lambda v: torch.from_numpy(np.ascontiguousarray(v)).to("cuda:0")  # noqa: E731
    r = up(p.rhs)
    x = torch.full_like(r, float("nan"))
    ref = prec != "tf32"
    h = B.kkt_analyze(p, B.kkt_default_options(prec, structured_s=s, max_refine=0 if ref else 10, refine_tol=1e-13))
    try:
        B.kkt_factor(h, up(p.a_vals), up(p.b_vals), up(p.c_vals))
        for _ in range(2):  # the second solve finds the first one's published vectors
            B.kkt_solve(h, r, x)
            eta = oracle.backward_error(p, x.cpu().numpy())
            assert eta <= (16 * (n + 2) * 2.0 ** -53 if ref else 1e-13), eta
    finally:
        B.kkt_destroy(h)


def test_solve_with_an_envelope_that_skips_blocks():
    """A row block of S that starts left of a row block above it: the products
    with the skipped blocks between them are zero."""
    torch = _torch()
    from dataclasses import replace

    import oracle
    from paper_1907_05420_gb300 import binding as B

    p = make_problem(GridSpec(5, 6, 2, 1, 3, 1e-1, 1e1, 7, "tiny"))
    n = 300
    rng = np.random.default_rng(5)
    cols = [[0, 200], [70, 290], [140, 150]]
    b_row = np.full(6, p.nA - 1, dtype=np.int32)
    p = replace(p, nC=n, c_vals=10.0 ** rng.uniform(-1, 1, n), b_blockptr=np.array([0, 2, 4, 6], np.int32), b_row=b_row,
                b_col=np.array(sum(cols, []), np.int32), b_vals=rng.standard_normal(6),
                rhs=rng.standard_normal(p.N * p.nA + n))
    up = lambda v: torch.from_numpy(np.ascontiguousarray(v)).to("cuda:0")  # noqa: E731
    xs = []
    for s in (0, 1):
        h = B.kkt_analyze(p, B.kkt_default_options("fp64", structured_s=s, max_refine=0, refine_tol=1e-14))
        try:
            r = up(p.rhs)
            x = torch.full_like(r, float("nan"))
            B.kkt_factor(h, up(p.a_vals), up(p.b_vals), up(p.c_vals))
            B.kkt_solve(h, r, x)
            xs.append(x.cpu().numpy())
        finally:
            B.kkt_destroy(h)
        assert oracle.backward_error(p, xs[-1]) <= 1e-14
    assert np.max(np.abs(xs[0] - xs[1])) <= 1e-10 * np.max(np.abs(xs[0]))
