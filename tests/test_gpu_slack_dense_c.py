"""kkt_slack_reduce with a dense C (its off-diagonal entries are copied, its
diagonal is written) against the oracle, bit for bit; A and C in place or not,
also one of them only, and a small grid beside a coupling wider than a block."""
from dataclasses import replace

import numpy as np
import pytest

from gen import CONFIGS, GridSpec, make_ipm_state, make_problem
from oracle import slack as oslack

pytestmark = pytest.mark.gpu

CASES = {"tiny_L4": (CONFIGS["tiny"], 4), "st5_n40_L4": (GridSpec(5, 6, 2, 4, 40, 1e-4, 1e4, 5, "st5"), 4)}


@pytest.mark.parametrize("in_place", [(0, 0), (0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize("case", sorted(CASES))
def test_reduce_with_dense_c(case, in_place):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_05420_gb300 import binding as B

    spec, L = CASES[case]
    p = make_problem(spec, flow_limits=L)
    st = make_ipm_state(p, 23)
    a_ref, c_diag, r_ref = oslack.slack_reduce(p, st)
    c = np.random.default_rng(3).standard_normal((p.nC, p.nC))
    c = c + c.T
    np.fill_diagonal(c, st.c_base)
    c_ref = c.copy()
    np.fill_diagonal(c_ref, c_diag)
    h = B.kkt_analyze(replace(p, c_kind=1, c_vals=c.reshape(-1).copy()))
    sl = B.Slack(h, p.ineq_rows)
    try:
        up = lambda v: torch.from_numpy(np.ascontiguousarray(v, dtype=np.float64)).to("cuda:0")  # noqa: E731
        state = {k: up(getattr(st, k)) for k in ("x", "z", "s", "y", "la", "le", "lcd", "lb", "lf")}
        a_base, c_base = up(st.a_base), up(c.reshape(-1))
        a_out = a_base if in_place[0] else torch.full_like(a_base, float("nan"))
        c_out = c_base if in_place[1] else torch.full_like(c_base, float("nan"))
        rhs = torch.full((p.nK,), float("nan"), dtype=torch.float64, device="cuda:0")
        sl.reduce(state, a_base, c_base, a_out, c_out, rhs)
        torch.cuda.synchronize()
    finally:
        sl.close()
        B.kkt_destroy(h)
    assert np.array_equal(a_out.cpu().numpy().reshape(p.N, -1), a_ref)
    assert np.array_equal(c_out.cpu().numpy().reshape(p.nC, p.nC), c_ref)
    assert np.array_equal(rhs.cpu().numpy(), r_ref)
