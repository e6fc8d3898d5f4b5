"""A handle's second kkt_solve takes about as long as its later ones: the graph
of the application is built by the first kkt_factor while the device is busy, not
inside a solve (which made the second solve of a small system 1.8 times as long as
the later ones).  The best of a dozen handles, so that the host's noise is out."""
import time

import numpy as np
import pytest

from gen import CONFIGS, make_problem

pytestmark = pytest.mark.gpu


def test_second_solve_pays_for_no_graph():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_05420_gb300 import binding as B

    p = make_problem(CONFIGS["grid30_n24"])
    up = lambda v: torch.from_numpy(np.ascontiguousarray(v)).to("cuda:0")  # noqa: E731
    vals, r = [up(v) for v in (p.a_vals, p.b_vals, p.c_vals)], up(p.rhs)
    x = torch.empty_like(r)
    times = []
    for _ in range(12):
        h = B.kkt_analyze(p, B.kkt_default_options("fp64", max_refine=0))
        try:
            B.kkt_factor(h, *vals)
            torch.cuda.synchronize()
            row = []
            for _ in range(8):
                t = time.perf_counter()
                B.kkt_solve(h, r, x, allow_not_converged=True)
                row.append(time.perf_counter() - t)
            times.append(row)
        finally:
            B.kkt_destroy(h)
    best = np.min(np.array(times), axis=0)
    assert best[1] <= 1.4 * best[2:].min(), best
