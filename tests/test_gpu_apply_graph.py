"""kkt_solve's host loop from graphs (use_graphs: from the second application and
the second refinement step of a kind of factor of S on) against direct launches:
the same solutions bit for bit, steps, eta and fallback, over repeated solves
with new right-hand sides, several at once, a new factor, and caller streams."""
from dataclasses import replace

import numpy as np
import pytest

from gen import CONFIGS, make_problem

pytestmark = pytest.mark.gpu


def _solves(torch, p, prec, graphs, opts):
    from paper_1907_05420_gb300 import binding as B

    rng = np.random.default_rng(5)
    rhs = [p.rhs, rng.standard_normal(p.nK), rng.standard_normal(p.nK) * 1e6, p.rhs]
    vals = [np.ascontiguousarray(v) for v in (p.a_vals, p.b_vals, p.c_vals)]
    h = B.kkt_analyze(p, B.kkt_default_options(prec, use_graphs=graphs, **opts))
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    out = []
    try:
        for turn in range(2):
            B.kkt_factor(h, *vals)
            torch.cuda.synchronize()  # the solves below may run on other streams
            for q, r in enumerate(rhs):
                x = np.empty(p.nK)
                B.kkt_solve(h, np.ascontiguousarray(r), x, allow_not_converged=True,
                            stream=streams[q % 2].cuda_stream if turn else 0)
                i = B.kkt_get_info(h)
                out.append((x, i["refine_steps"], i["rel_residual"], i["fell_back_fp64"]))
            many = np.ascontiguousarray(np.stack(rhs))
            x = np.empty_like(many)
            B.kkt_solve(h, many, x, nrhs=len(rhs), allow_not_converged=True)
            out.append((x, 0, 0.0, 0))
    finally:
        B.kkt_destroy(h)
    return out


@pytest.mark.parametrize("name,prec,opts", [
    ("grid30_n24", "fp64", {}),
    ("grid30_n24", "fp64", {"refine_tol": 0.0, "max_refine": 4}),
    ("grid30_n24", "fp64", {"early_solve": 1}),
    ("grid30_n24", "fp64", {"structured_s": 2}),
    ("grid30_n24", "fp64", {"refine_mode": 1, "refine_tol": 1e-17}),
    ("grid2383_n6", "tf32", {"refine_tol": 1e-13}),
    ("grid2383_n6", "bf16", {"refine_tol": 1e-13}),
])
def test_graph_equals_direct(name, prec, opts):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    spec = replace(CONFIGS["grid2383_n96"], n_per=6) if name == "grid2383_n6" else CONFIGS[name]
    p = make_problem(spec, coupling="paper") if opts.get("structured_s") else make_problem(spec)
    direct, graph = (_solves(torch, p, prec, g, opts) for g in (0, 1))
    for q, ((x0, s0, e0, f0), (x1, s1, e1, f1)) in enumerate(zip(direct, graph)):
        assert np.array_equal(x0, x1) and (s0, e0, f0) == (s1, e1, f1), q
