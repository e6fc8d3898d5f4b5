"""The dense tails' update by their heavy descendants (one emulated-FP64
product per tail) against the plain FP64 path, whose supernodal kernel applies
the same updates: grids with many meshes, so that supernodes below the tail
reach a large part of its rows; few and many periods, ragged tail orders.  Both
are refined to eta <= 1e-15 with their own factors; with a barrier over six
decades the solutions then agree to 1e-9, and a lost or misplaced update would
leave a factor that refinement cannot use (the inertia would change too)."""
import numpy as np
import pytest

from gen import GridSpec, make_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("spec", [
    GridSpec(700, 1300, 105, 40, 3, 1e-3, 1e3, 5),
    GridSpec(1500, 2300, 225, 33, 5, 1e-3, 1e3, 6),
    GridSpec(2383, 2900, 327, 100, 2, 1e-3, 1e3, 7),
    GridSpec(901, 1801, 130, 1, 1, 1e-3, 1e3, 8),
], ids=lambda s: f"{s.n_bus}x{s.n_per}")
def test_heavy_update_matches_fp64(spec):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    from paper_1907_05420_gb300 import binding as B

    p = make_problem(spec)
    xs = {}
    for prec in ("fp64", "f64emu"):
        s = B.KKTSolver(p, prec, refine_tol=1e-15, structured_s=1)
        s.factor()
        xs[prec] = s.solve()
        info = s.info()
        s.close()
        assert info["dense_tail_cols"] >= 512
        assert [info["n_pos"], info["n_neg"], info["n_zero"]] == [p.N * p.nP + p.nC, p.N * (p.nA - p.nP), 0]
        assert oracle.backward_error(p, xs[prec]) <= 1e-15
    assert np.max(np.abs(xs["f64emu"] - xs["fp64"])) <= 1e-9 * np.max(np.abs(xs["fp64"]))
