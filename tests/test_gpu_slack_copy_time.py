"""kkt_slack_reduce with a dense C that is not in place moves C at the memory's
rate: it takes at most six times as long as device copies of the same A and C (its
other work is a fraction of theirs at this size; a loop that a few CTAs run takes
twenty times as long)."""
from dataclasses import replace

import numpy as np
import pytest

from gen import GridSpec, make_ipm_state, make_problem

pytestmark = pytest.mark.gpu


def test_dense_c_is_copied_at_memory_rate():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_05420_gb300 import binding as B

    p = make_problem(GridSpec(1100, 1400, 45, 1000, 4, 1e-3, 1e3, 7), flow_limits=200)
    st = make_ipm_state(p, 23)
    c = np.random.default_rng(3).standard_normal((p.nC, p.nC))
    h = B.kkt_analyze(replace(p, c_kind=1, c_vals=c.reshape(-1)))
    sl = B.Slack(h, p.ineq_rows)
    try:
        up = lambda v: torch.from_numpy(np.ascontiguousarray(v, dtype=np.float64)).to("cuda:0")  # noqa: E731
        state = {k: up(getattr(st, k)) for k in ("x", "z", "s", "y", "la", "le", "lcd", "lb", "lf")}
        a_base, c_base = up(st.a_base), up(c.reshape(-1))
        a_out, c_out = torch.empty_like(a_base), torch.empty_like(c_base)
        rhs = torch.empty(p.nK, dtype=torch.float64, device="cuda:0")

        def best(f):
            ts = []
            for _ in range(20):
                e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
                e[0].record()
                f()
                e[1].record()
                torch.cuda.synchronize()
                ts.append(e[0].elapsed_time(e[1]))
            return min(ts)

        def copies():
            a_out.copy_(a_base)
            c_out.copy_(c_base)

        t_copy = best(copies)
        t_reduce = best(lambda: sl.reduce(state, a_base, c_base, a_out, c_out, rhs))
    finally:
        sl.close()
        B.kkt_destroy(h)
    assert t_reduce <= 6 * t_copy, (t_reduce, t_copy)
    off = ~np.eye(p.nC, dtype=bool)
    assert np.array_equal(c_out.cpu().numpy().reshape(p.nC, p.nC)[off], c[off])
