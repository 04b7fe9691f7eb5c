"""The scaled entries in their place in the layout: short rows copied by a few lanes each, long rows
by a warp per chunk of 256 entries, at the edges of both (128 entries make a row long; chunks one
entry short, full and one over; a dense row and column among short ones), in the three value types.

FP64: iterates against the oracle at the repository's 1e-10.  BF16: +-1 coefficients are exact under
the power-of-two scaling, so the run equals the FP32 one bit for bit.  FP32: before a restart the
iterates follow FP64 to the repository's 1e-5."""
import numpy as np
import pytest

from oracle import rhpdhg_oracle as O
from paper_2407_16144_gb300 import lpgen

pytestmark = pytest.mark.gpu

LENGTHS = {
    "chunk_edges": [127, 128, 129, 255, 256, 257, 511, 512, 513, 0, 1, 3, 1024, 1025] * 3,
    "dense_row": [2] * 500 + [2000] + [2] * 533,
    "all_long": [150 + i for i in range(70)],
    "mean_over_32": [40] * 63 + [128] * 2 + [300],
}


@pytest.fixture(scope="module")
def rh():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2407_16144_gb300 import _build, rhpdhg
    _build.build()
    rhpdhg.load()
    return rhpdhg


def _lp(name, transpose):
    rng = np.random.default_rng(31)
    lens = np.asarray(LENGTHS[name])
    k, width = len(lens), 2000
    rows = np.repeat(np.arange(k), lens)
    cols = np.concatenate([rng.choice(width, n, replace=False) for n in lens])
    m, n = (width, k) if transpose else (k, width)
    if transpose:
        rows, cols = cols, rows
    rp, ci, val = lpgen.coo_to_csr(m, n, rows, cols, rng.choice([-1.0, 1.0], len(rows)))
    return lpgen.LP(m_eq=m // 2, m_ineq=m - m // 2, n=n, row_ptr=rp, col_idx=ci, val=val,
                    c=rng.standard_normal(n), q=rng.standard_normal(m),
                    l=rng.uniform(-2.0, 0.0, n), u=rng.uniform(0.5, 3.0, n))


def _run(rh, lp, T, **kw):
    with rh.Solver(lp, algorithm=1, eps_rel_kkt=1e-14, max_iters=T, first_epoch_len=100,
                   check_every=16, **kw) as s:
        s.run()
        return s.state(1)


@pytest.mark.parametrize("transpose", [False, True], ids=["rows", "columns"])
@pytest.mark.parametrize("name", list(LENGTHS))
def test_entries_of_short_and_long_rows(rh, name, transpose):
    lp, T = _lp(name, transpose), 40
    f64 = _run(rh, lp, T)
    o = O.solve(lp, O.OracleParams(algorithm=1, eps_rel_kkt=1e-14, max_iters=T,
                                   first_epoch_len=100, check_every=16), snapshot_iters=[T - 1])
    snap = o.snapshots[T - 1]
    for got, want in zip(f64, (snap["xt"], snap["yt"])):
        assert np.abs(got - want).max() <= 1e-10 * max(1.0, np.abs(want).max())
    for got, want in zip(_run(rh, lp, T, precision=1), f64):
        assert np.abs(got - want).max() <= 1e-5 * max(1.0, np.abs(want).max())
    for got, want in zip(_run(rh, lp, T, precision=2),
                         _run(rh, lp, T, precision=1, pow2_scaling=1)):
        assert np.array_equal(got, want)
