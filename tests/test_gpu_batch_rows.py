"""The batched kernel's row products over every group width it may take (1 to 32 threads a row, by
the mean row length), rows longer than the entries it keeps in flight, row counts around a warp's
32 rows and the CTA's 512 threads, against the oracle in FP64 (mixed slots run the same template):
1e-10 in the max norm after 60 iterations with restarts, the repository's tolerance."""
import numpy as np
import pytest

from oracle import rhpdhg_oracle as O
from paper_2407_16144_gb300 import lpgen, rhpdhg as rh

pytestmark = pytest.mark.gpu


def _skewed(m, n):
    """Rows of 1 to 60 entries around a mean of six, one dense row."""
    rng = np.random.default_rng(31)
    lens = np.minimum(np.minimum(rng.zipf(1.7, m) + 1, 60), n)
    lens[m // 2] = n
    rp = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    col = np.concatenate([np.sort(rng.choice(n, k, replace=False)) for k in lens])
    return lpgen.LP(m_eq=m // 2, m_ineq=m - m // 2, n=n, row_ptr=rp, col_idx=col.astype(np.int32),
                    val=rng.uniform(0.5, 2.0, rp[-1]) * rng.choice([-1.0, 1.0], rp[-1]),
                    c=rng.standard_normal(n), q=rng.standard_normal(m), l=np.zeros(n),
                    u=np.where(rng.random(n) < 0.3, 2.0, np.inf))


LPS = {
    "groups_1_1": lambda: lpgen.make_standard_planted(1, m=90, n=100, col_nnz=1),
    "groups_4_2": lambda: lpgen.make_standard_planted(2, m=129, n=323, col_nnz=3),
    "groups_8_4": lambda: lpgen.make_standard_planted(3, m=33, n=80, col_nnz=5),
    "groups_16_8": lambda: lpgen.make_standard_planted(4, m=200, n=513, col_nnz=10),
    "groups_32_16": lambda: lpgen.make_standard_planted(5, m=100, n=260, col_nnz=25),
    "groups_32_32": lambda: lpgen.make_standard_planted(6, m=512, n=1025, col_nnz=80),
    "skewed": lambda: _skewed(511, 700),
}


@pytest.mark.parametrize("name", list(LPS))
def test_batch_rows_match_oracle(name):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2407_16144_gb300 import _build
    _build.build()
    lp = LPS[name]()
    common = dict(algorithm=1, eps_rel_kkt=1e-14, max_iters=60, first_epoch_len=20, check_every=16)
    o = O.solve(lp, O.OracleParams(**common))
    need = rh.rhpdhg_batch_bytes_needed(rh.host_problem(lp, []), 0)
    with rh.Batch(2, 2 * need + (1 << 16)) as b:
        slots = [b.add(lp, **common) for _ in range(2)]
        res = b.run_all(slots, iters=7)
    for s in slots:
        r = res[s]
        assert r.iters == 60
        for got, want in ((r.x, o.x), (r.y, o.y)):
            assert np.abs(got - want).max() <= 1e-10 * max(1.0, np.abs(want).max())
    assert np.array_equal(res[slots[0]].x, res[slots[1]].x)
