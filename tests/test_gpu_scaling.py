"""The diagonal scalings over their parameters: numbers of Ruiz passes that end in either of the two
pairs of buffers the passes go between (0, 1, 2, 3, 10), Pock-Chambolle left out (alpha < 0), as a sum
(1) and as sums of powers (0.5, 1.5), on LPs whose mean row lengths take each number of lanes per row,
with long, empty and single-entry rows and ragged sizes on either side; single LPs and batched slots.

Tolerance against the oracle: a pass turns a factor f and its row's statistic into f / sqrt(stat),
where the factors' own errors average out, so that each pass adds a few roundings (8 allowed), a sum
at most its number of terms, a power's or square root's own error less than 16; twice that, both
sides rounding: 2 (8 passes + longest row + 16) 2^-53.  Iterates: the repository's 1e-10."""
import numpy as np
import pytest

from oracle import rhpdhg_oracle as O
from paper_2407_16144_gb300 import lpgen

pytestmark = pytest.mark.gpu

rng0 = np.random.default_rng(11)
LENGTHS = {
    "mean_2": [0, 1, 3, 2] * 97 + [40, 33, 1],           # over 32 entries: a long row of one lane
    "mean_6": [6, 5, 7, 0, 1] * 40 + [300] + [6] * 60,
    "mean_12": list(rng0.integers(0, 25, size=231)),
    "mean_24": [24] * 100 + [700, 1, 0] + [20] * 30,
    "mean_50": [50, 51, 49, 0] * 20 + [513],
    "mean_100": [100] * 33 + [0, 1, 400],
    "mean_300": [300, 299, 310, 1200] * 9 + [0, 1],
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
    rng = np.random.default_rng(37)
    lens = np.asarray(LENGTHS[name])
    k, width = len(lens), 1500
    rows = np.repeat(np.arange(k), lens)
    cols = np.concatenate([rng.choice(width, n, replace=False) for n in lens]).astype(np.int64)
    m, n = (width, k) if transpose else (k, width)
    if transpose:
        rows, cols = cols, rows
    val = np.exp(rng.standard_normal(len(rows))) * rng.choice([-1.0, 1.0], len(rows))
    rp, ci, val = lpgen.coo_to_csr(m, n, rows, cols, val)
    return lpgen.LP(m_eq=m // 2, m_ineq=m - m // 2, n=n, row_ptr=rp, col_idx=ci, val=val,
                    c=rng.standard_normal(n), q=rng.standard_normal(m),
                    l=rng.uniform(-2.0, 0.0, n), u=rng.uniform(0.5, 3.0, n))


@pytest.mark.parametrize("ruiz", [0, 1, 2, 3, 10])
@pytest.mark.parametrize("alpha", [-1.0, 0.5, 1.0, 1.5])
def test_scaling_parameters_match_oracle(rh, ruiz, alpha):
    for name in LENGTHS:
        for transpose in (False, True):
            lp = _lp(name, transpose)
            A = O.csr_matrix(lp)
            _, Do, Eo = O.scale_problem(A, ruiz, alpha)
            with rh.Solver(lp, ruiz_iters=ruiz, pock_chambolle_alpha=alpha, power_iters=1) as s:
                D, E = s.scaling()[:2]
            longest = max(np.diff(A.indptr).max(), np.diff(A.tocsc().indptr).max())
            tol = 2 * (8 * (ruiz + 1) + longest + 16) * 2.0 ** -53
            for got, want in ((D, Do), (E, Eo)):
                assert np.abs(got / want - 1.0).max() <= tol, (name, transpose)


@pytest.mark.parametrize("ruiz, alpha", [(0, -1.0), (0, 1.0), (3, -1.0), (3, 0.5), (2, 1.5)])
def test_batched_slot_scaling_parameters(rh, ruiz, alpha):
    lps = [lpgen.make_standard_planted(seed=2, m=90, n=230), lpgen.make_tiny_general(3, 3, 4, 9),
           lpgen.make_c2(7, scale=0.004)]            # feasible: no certificate ends them early
    T = 60
    common = dict(algorithm=1, eps_rel_kkt=1e-14, max_iters=T, check_every=16, first_epoch_len=20)
    with rh.Batch(4, 64 << 20) as b:
        slots = [b.add(lp, ruiz_iters=ruiz, pock_chambolle_alpha=alpha, **common) for lp in lps]
        res = b.run_all(slots, iters=40)
    for lp, s in zip(lps, slots):
        o = O.solve(lp, O.OracleParams(ruiz_iters=ruiz, pock_chambolle_alpha=alpha, **common))
        for got, want in ((res[s].x, o.x), (res[s].y, o.y)):
            assert np.abs(got - want).max() <= 1e-10 * max(1.0, np.abs(want).max())
