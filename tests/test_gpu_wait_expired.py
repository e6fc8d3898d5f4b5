"""What a bounded device wait that runs out leaves behind (set by the diagnostic
call; no wait is made to run out): the next call that reads results on the host
says so, in the whole solve and in the steps of a distributed one, and the next
factorization clears it."""
import numpy as np
import pytest

from gen import CONFIGS, make_problem

pytestmark = pytest.mark.gpu

KKT_ERR_TIMEOUT = 7


def _torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


@pytest.mark.parametrize("graphs", [0, 1])
def test_solve_reports_it_until_the_next_factor(graphs):
    _torch()
    import oracle
    from paper_1907_05420_gb300 import binding as B

    p = make_problem(CONFIGS["grid30_n24"])
    s = B.KKTSolver(p, "fp64", use_graphs=graphs)
    try:
        for _ in range(3):
            s.factor()
            assert oracle.backward_error(p, s.solve()) <= 1e-10
            B.kkt_probe_wait_expired(s.h)
            for _ in range(2):
                with pytest.raises(B.KKTError) as e:
                    s.solve()
                assert e.value.status == KKT_ERR_TIMEOUT
    finally:
        s.close()


def test_the_steps_of_a_distributed_solve_report_it():
    _torch()
    from paper_1907_05420_gb300 import binding as B
    from paper_1907_05420_gb300.sharded import GpuShard, shard_of

    p = make_problem(CONFIGS["grid30_n24"])
    be = GpuShard(shard_of(p, 0, p.N, True))
    try:
        for _ in range(2):
            be.factor(p.a_vals, p.b_vals, p.c_vals)
            be.factor_schur()
            r = be.upload(p.rhs)
            x = be.back(be.coupling_solve(be.front(r)), 0, p.nC)
            assert np.isfinite(be.norm(x, 0, x.numel()))
            B.kkt_probe_wait_expired(be.h)
            x = be.back(be.coupling_solve(be.front(r)), 0, p.nC)
            with pytest.raises(B.KKTError) as e:
                be.norm(be.residual(r, x), 0, x.numel())
            assert e.value.status == KKT_ERR_TIMEOUT
    finally:
        be.close()
