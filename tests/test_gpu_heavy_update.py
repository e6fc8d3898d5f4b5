"""The dense tails' update by their heavy descendants as one emulated product,
where it really runs: the host analysis says for every grid which supernodes it
takes (one grid comes close to the 256 columns it holds).

One application of the factors, without refinement, has the backward error of the
plain FP64 path up to the emulation's own: a product of 256 columns is off by at
most 256 roundings of its largest term, and an FP64 factor's error is at least
one rounding of it.

A NaN in a heavy panel's row of the tail makes that row of the tail NaN, as in
FP64 products: its diagonal entry stays NaN until it is a pivot, and this pivot
and the later ones of its 64-column diagonal block are counted as zero."""
import numpy as np
import pytest

from gen import GridSpec, make_problem
from test_symbolic import C, _lib, _ptr

SPECS = [
    GridSpec(901, 1801, 130, 1, 1, 1e-3, 1e3, 8),
    GridSpec(1200, 2600, 180, 36, 2, 1e-3, 1e3, 6),
    GridSpec(1500, 2300, 225, 33, 5, 1e-3, 1e3, 6),
    GridSpec(7000, 12000, 1050, 210, 1, 1e-3, 1e3, 5),
]


def heavy(p):
    """The emulated tail's analysis: its heavy supernodes and the arrays below."""
    L = _lib()
    i32 = [np.ascontiguousarray(v, dtype=np.int32) for v in (p.a_rowptr, p.a_col, p.b_blockptr, p.b_row, p.b_col)]
    hint = np.ascontiguousarray(np.asarray(p.a_vals).reshape(p.N, -1)[0], dtype=np.float64)
    rp, col, bbp, brow, bcol = (_ptr(v, C.c_int32) for v in i32)
    h = L.kkt_symbolic_create(p.nA, p.nP, rp, col, _ptr(hint, C.c_double), p.N, p.nC, bbp, brow, bcol, int(p.c_kind))
    try:
        nT = L.kkt_symbolic_choose_tail(h, 1.5, 96 << 30)
        out = {"tail_col": p.nA - nT}
        for name in ("heavy", "sn_first", "sn_rowptr", "sn_rows", "sn_valoff", "a_map"):
            a = np.zeros(L.kkt_symbolic_get(h, name.encode(), None), dtype=np.int64)
            L.kkt_symbolic_get(h, name.encode(), _ptr(a, C.c_int64))
            out[name] = a
    finally:
        L.kkt_symbolic_destroy(h)
    return out


def columns(p):
    s = heavy(p)
    assert p.nA - s["tail_col"] >= 512
    return int((s["sn_first"][s["heavy"] + 1] - s["sn_first"][s["heavy"]]).sum())


# few coupling columns, whose pivots may be NaN too
NAN_SPECS = [SPECS[0], GridSpec(1200, 2600, 180, 1, 2, 1e-3, 1e3, 6), GridSpec(1500, 2700, 225, 2, 3, 1e-3, 1e3, 5)]


def nan_entry(p):
    """(pivots it must make NaN, entry of A) for an entry in a tail row of a heavy
    panel with no row outside the tail but its own columns: nothing else carries
    the entry to the tail."""
    s = heavy(p)
    nT = p.nA - s["tail_col"]
    best = (0, -1)
    for q in s["heavy"]:
        w, rows = s["sn_first"][q + 1] - s["sn_first"][q], s["sn_rows"][s["sn_rowptr"][q]:s["sn_rowptr"][q + 1]]
        if rows[w] < s["tail_col"]:
            continue
        at = s["a_map"] - s["sn_valoff"][q]
        for e in np.nonzero((at >= 0) & (at < w * len(rows)) & (at % len(rows) >= w))[0]:
            row = rows[at[e] % len(rows)] - s["tail_col"]
            best = max(best, (min(64 - row % 64, nT - row), e))
    return best


def test_specs_have_heavy_descendants():
    cols = [columns(make_problem(s)) for s in SPECS]
    assert all(0 < c <= 256 for c in cols) and max(cols) > 240, cols
    for p in map(make_problem, NAN_SPECS):
        assert nan_entry(p)[0] > p.nC


def _torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


@pytest.mark.gpu
@pytest.mark.parametrize("spec", SPECS, ids=lambda s: f"{s.n_bus}x{s.n_per}")
def test_one_application(spec):
    _torch()
    import oracle
    from paper_1907_05420_gb300 import binding as B

    p = make_problem(spec)
    eta = {}
    for prec in ("fp64", "f64emu"):
        s = B.KKTSolver(p, prec, structured_s=1, max_refine=0)
        s.factor()
        x = s.solve(allow_not_converged=True)
        info = s.info()
        s.close()
        assert [info["n_pos"], info["n_neg"], info["n_zero"]] == [p.N * p.nP + p.nC, p.N * (p.nA - p.nP), 0]
        eta[prec] = oracle.backward_error(p, x)
    assert eta["f64emu"] <= 256 * max(eta["fp64"], 2.0 ** -53), eta


@pytest.mark.gpu
@pytest.mark.parametrize("spec", NAN_SPECS, ids=lambda s: f"{s.n_bus}x{s.n_per}")
def test_nan_in_a_heavy_panel_reaches_the_tail(spec):
    _torch()
    from paper_1907_05420_gb300 import binding as B

    p = make_problem(spec)
    zeros, entry = nan_entry(p)
    a = np.array(p.a_vals, dtype=np.float64).reshape(p.N, -1)
    a[p.N // 2, entry] = np.nan
    s = B.KKTSolver(p, "f64emu", structured_s=1)
    try:
        for _ in range(2):  # the second time as a graph, after a factor of finite panels
            s.factor(a_vals=a)
            info = s.info()
            assert info["n_zero"] >= zeros, (info, zeros)
            with pytest.raises(B.KKTError) as err:
                s.solve()
            assert err.value.status == 9  # KKT_ERR_NONFINITE
            s.factor()
            s.solve()
            assert s.info()["n_zero"] == 0
    finally:
        s.close()
