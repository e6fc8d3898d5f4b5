"""The block factor's panels (small ones by eight lanes, larger ones by their
triangle and rows, the longest split over CTAs) with the dense tail off, which
puts the whole elimination tree through them, against the dense tail: grids whose
panels go from one column to 32 columns and beyond 256 rows, few and many blocks.
Both are refined to eta <= 1e-15 with their own factors (the solutions then agree
to 1e-9), with the inertia of a quasi-definite K; with a threshold that perturbs
pivots (not refined to the target: the inertia alone), the counts agree."""
import numpy as np
import pytest

from gen import CONFIGS, GridSpec, make_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "f64emu"])
@pytest.mark.parametrize("spec", [
    CONFIGS["tiny"],
    GridSpec(30, 41, 6, 3, 37, 1e-3, 1e3, 4),
    GridSpec(301, 411, 40, 13, 3, 1e-3, 1e3, 5),
    GridSpec(901, 1801, 130, 1, 2, 1e-3, 1e3, 6),
    GridSpec(2383, 2900, 327, 100, 1, 1e-3, 1e3, 7),
], ids=lambda s: f"{s.n_bus}x{s.n_per}")
def test_panels_match_dense_tail(spec, prec):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    from paper_1907_05420_gb300 import binding as B

    p = make_problem(spec)
    xs, counts = [], []
    for tail in (0, 1):
        s = B.KKTSolver(p, prec, refine_tol=1e-15, dense_tail=tail)
        s.factor()
        xs.append(s.solve())
        info = s.info()
        s.close()
        assert [info["n_pos"], info["n_neg"], info["n_zero"]] == [p.N * p.nP + p.nC, p.N * (p.nA - p.nP), 0]
        assert oracle.backward_error(p, xs[-1]) <= 1e-15
        s = B.KKTSolver(p, prec, pivot_eps=1e-4, dense_tail=tail)
        s.factor()
        s.solve(allow_not_converged=True)
        info = s.info()
        s.close()
        counts.append([info[k] for k in ("n_pos", "n_neg", "n_zero", "n_perturbed")])
    assert np.max(np.abs(xs[0] - xs[1])) <= 1e-9 * np.max(np.abs(xs[1]))
    assert counts[0] == counts[1]


@pytest.mark.parametrize("spec", [CONFIGS["tiny"], GridSpec(301, 411, 40, 13, 3, 1e-3, 1e3, 5)],
                         ids=lambda s: f"{s.n_bus}x{s.n_per}")
def test_threshold_that_is_not_positive(spec):
    """pivot_eps = 0 turns the perturbation off, also where max|A_i| is infinite
    (0 * Inf is no threshold)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_05420_gb300 import binding as B

    p = make_problem(spec)
    a = np.array(p.a_vals, dtype=np.float64).reshape(p.N, -1)
    a[0, 0] = np.inf
    for tail in (0, 1):
        h = B.kkt_analyze(p, B.kkt_default_options("fp64", pivot_eps=0.0, dense_tail=tail))
        try:
            B.kkt_factor(h, a, np.ascontiguousarray(p.b_vals), np.ascontiguousarray(p.c_vals))
            assert B.kkt_get_info(h)["n_perturbed"] == 0
        finally:
            B.kkt_destroy(h)
