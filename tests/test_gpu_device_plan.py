"""The layout planned on the device (k_plan_tiles, k_plan_scan, k_plan_emit) at the edges of its
tiles (32 rows), its blocks (64 tiles) and its branches: its summary equals the host plan's
(rhpdhg_plan_layout), and the products and iterates that walk it equal the oracle's.

The iterates' tolerance is the repository's for FP64 handles: 1e-10 in the max norm."""
import numpy as np
import pytest

from oracle import rhpdhg_oracle as O
from paper_2407_16144_gb300 import lpgen

pytestmark = pytest.mark.gpu

rng0 = np.random.default_rng(5)
LENGTHS = {
    "one_row": [3],
    "31_rows": [4] * 31,
    "33_rows": [0] + [4] * 32,
    "64_tiles": [2] * (64 * 32),
    "64_tiles_and_a_row": [2] * (64 * 32) + [5],
    "130_tiles_mixed": list(rng0.integers(0, 30, size=130 * 32 - 7)),
    "long_by_length": [129, 1, 300, 2000, 0, 128] * 30,
    "budget_ties": [40] * 32 * 5 + [1] * 9,
    "budget_two_leave": [100] * 12 + [0] * 20 + [128] * 9 + [3] * 23,
    "long_in_every_block": ([1] * 31 + [700]) * 70,
    "single_entries_ragged": [1] * 4001,
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


def _lp(lens):
    rng = np.random.default_rng(29)
    lens = np.asarray(lens, dtype=np.int64)
    m, n = len(lens), max(2100, len(lens) // 2)
    rp = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    col = np.concatenate([np.sort(rng.choice(n, k, replace=False)) for k in lens])
    m_eq = m // 2
    return lpgen.LP(m_eq=m_eq, m_ineq=m - m_eq, n=n, row_ptr=rp, col_idx=col.astype(np.int32),
                    val=rng.uniform(0.5, 2.0, rp[-1]) * rng.choice([-1.0, 1.0], rp[-1]),
                    c=rng.standard_normal(n), q=rng.standard_normal(m),
                    l=np.where(rng.random(n) < 0.5, 0.0, -np.inf),
                    u=np.where(rng.random(n) < 0.3, 2.0, np.inf))


@pytest.mark.parametrize("name", list(LENGTHS))
def test_device_plan_and_products(rh, name):
    lp = _lp(LENGTHS[name])
    A = O.csr_matrix(lp)
    common = dict(algorithm=1, eps_rel_kkt=1e-14, max_iters=60, first_epoch_len=20, check_every=16)
    with rh.Solver(lp, **common) as s:
        lay = s.layout()
        r = s.run()
        xt, yt = s.state(1)
    for side, ptr in (("row", A.indptr), ("col", A.T.tocsr().indptr)):
        rc, pl = rh.rhpdhg_plan_layout(ptr)
        assert rc == 0
        for dev, host in (("tile_mult", "tile_mult"), ("long_rows", "long_rows"),
                          ("chunks", "chunks"), ("seg", "seg"), ("wide_rows", "wide_rows")):
            assert lay[f"{dev}_{side}"] == pl[host], (side, dev, lay, pl)
    o = O.solve(lp, O.OracleParams(**common), snapshot_iters=[59])
    snap = o.snapshots[59]
    assert r.iters == 60
    for got, want in ((xt, snap["xt"]), (yt, snap["yt"])):
        assert np.abs(got - want).max() <= 1e-10 * max(1.0, np.abs(want).max())
