"""One application of a block factor whose whole elimination tree goes through the
supernodal panels (dense tail off), without refinement: its backward error against
the one with the dense tail.  Both factors are FP64 sums of the same products in
other orders; 16 times the larger of the tail's error and one rounding leaves room
for the order, and shows a factor that is digits worse."""
import pytest

from gen import CONFIGS, GridSpec, make_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("spec", [
    CONFIGS["tiny"],
    GridSpec(30, 41, 6, 3, 37, 1e-3, 1e3, 4),
    GridSpec(301, 411, 40, 13, 3, 1e-3, 1e3, 5),
    GridSpec(901, 1801, 130, 1, 2, 1e-3, 1e3, 6),
    GridSpec(2383, 2900, 327, 100, 1, 1e-3, 1e3, 7),
], ids=lambda s: f"{s.n_bus}x{s.n_per}")
def test_one_application(spec):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    from paper_1907_05420_gb300 import binding as B

    p = make_problem(spec)
    eta = []
    for tail in (0, 1):
        s = B.KKTSolver(p, "fp64", max_refine=0, dense_tail=tail)
        s.factor()
        eta.append(oracle.backward_error(p, s.solve(allow_not_converged=True)))
        s.close()
    assert eta[0] <= 16 * max(eta[1], 2.0 ** -53), eta
