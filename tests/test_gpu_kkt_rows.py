"""rhpdhg_kkt_eval's row kernel where its warps' segments begin, end and split: row counts around a
multiple of the 32 rows a warp takes, empty rows, rows around and beyond the entries a warp stages
at a time, and many entries in one of 32 rows.  Compared with numpy; every output's tolerance is
twice the bound of recursive FP64 summation, (terms) u sum |terms|, carried to that output."""
import numpy as np
import pytest

from paper_2407_16144_gb300 import lpgen

pytestmark = pytest.mark.gpu

STAGE = 704      # entries a warp stages at a time
LENGTHS = {
    "one_row": [3],
    "empty_rows_only": [0] * 33,
    "ragged_tiles": [5] * 31 + [0] + [7] * 33 + [1],
    "stage_edges": [STAGE - 1, 1, STAGE, 1, STAGE + 1, 0, 2 * STAGE, 3] + [1] * 60,
    "one_long_of_32": [0] * 7 + [5000] + [2] * 24 + [1] * 5,
    "even_rows": [22] * 32 * 9,                      # 704 per warp: one full stage
    "uneven_rows": [1, 40] * 400 + [128, 0, 0],
}


@pytest.mark.parametrize("name", list(LENGTHS))
def test_kkt_rows_match_numpy(name):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2407_16144_gb300 import _build, rhpdhg as rh
    _build.build()
    lens = np.asarray(LENGTHS[name], dtype=np.int64)
    rng = np.random.default_rng(23)
    m, n = len(lens), 6007
    rp = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    col = np.concatenate([np.sort(rng.choice(n, k, replace=False)) for k in lens] or [[]])
    val = rng.standard_normal(rp[-1])
    lp = lpgen.LP(m_eq=m // 2, m_ineq=m - m // 2, n=n, row_ptr=rp, col_idx=col.astype(np.int32),
                  val=val, c=rng.standard_normal(n), q=rng.standard_normal(m),
                  l=np.where(rng.random(n) < 0.5, 0.0, -np.inf),
                  u=np.where(rng.random(n) < 0.5, 2.0, np.inf))
    x, y = rng.uniform(0, 2, n), np.abs(rng.standard_normal(m))

    rows = np.repeat(np.arange(m), lens)
    cols = col.astype(np.int64)
    kx = np.bincount(rows, val * x[cols], m)
    ky = np.bincount(cols, val * y[rows], n)
    r = lp.q - kx
    r[lp.m_eq:] = np.maximum(r[lp.m_eq:], 0.0)
    g = lp.c - ky
    lf, uf = np.isfinite(lp.l), np.isfinite(lp.u)
    lam = np.where(lf & uf, g, np.where(lf, np.maximum(g, 0), np.where(uf, np.minimum(g, 0), 0)))
    at = np.where(lam > 0, lp.l, np.where(lam < 0, lp.u, 0.0))
    bnd = np.where(lam != 0, at * lam, 0.0)
    qn, cn = 1 + np.linalg.norm(lp.q), 1 + np.linalg.norm(lp.c)
    p, d = lp.c @ x, lp.q @ y + bnd.sum()
    want = [np.linalg.norm(r) / qn, np.linalg.norm(g - lam) / cn,
            abs(p - d) / (1 + abs(p) + abs(d)), p, d]

    eps = 2.0 ** -53
    er = (lens + 2) * eps * (np.bincount(rows, np.abs(val * x[cols]), m) + np.abs(lp.q))
    cnt = np.bincount(cols, minlength=n) + 2
    eg = cnt * eps * (np.bincount(cols, np.abs(val * y[rows]), n) + np.abs(lp.c))
    ep = (n + 1) * eps * np.abs(lp.c * x).sum()
    ed = ((m + 1) * eps * np.abs(lp.q * y).sum() + (n + 1) * eps * np.abs(bnd).sum()
          + (np.where(np.isfinite(at), np.abs(at), 0.0) * eg).sum())
    rel = (m + n) * eps
    tol = [2 * (np.linalg.norm(er) / qn + rel * want[0]), 2 * (np.linalg.norm(eg) / cn + rel * want[1]),
           2 * (2 * (ep + ed) / (1 + abs(p) + abs(d)) + rel), 2 * ep, 2 * ed]

    dev = lpgen.LP(**{f: (torch.as_tensor(getattr(lp, f), device="cuda")
                          if isinstance(getattr(lp, f), np.ndarray) else getattr(lp, f))
                      for f in ("m_eq", "m_ineq", "n", "row_ptr", "col_idx", "val", "c", "q", "l",
                                "u")})
    xd, yd = torch.as_tensor(x, device="cuda"), torch.as_tensor(y, device="cuda")
    rc, got = rh.rhpdhg_kkt_eval(rh.device_problem(dev), xd.data_ptr(), yd.data_ptr())
    assert rc == rh.OK, rh.rhpdhg_last_error(None)
    for a, b, t in zip(got, want, tol):
        assert abs(a - b) <= t, (got, want, tol)


def test_kkt_scratch_stays_in_the_buffer_cache():
    """n + 8200 doubles after the first call, no more after the second, given back on request."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2407_16144_gb300 import _build, rhpdhg as rh
    _build.build()
    rh.load()
    n = 1000
    f64 = dict(dtype=torch.float64, device="cuda")
    lp = lpgen.LP(m_eq=1, m_ineq=0, n=n, row_ptr=torch.tensor([0, 1], device="cuda"),
                  col_idx=torch.zeros(1, dtype=torch.int32, device="cuda"), val=torch.ones(1, **f64),
                  c=torch.ones(n, **f64), q=torch.ones(1, **f64), l=torch.zeros(n, **f64),
                  u=torch.ones(n, **f64))
    x, y = torch.ones(n, **f64), torch.ones(1, **f64)
    rh.release_cached_memory()
    for _ in range(2):
        rc, out = rh.rhpdhg_kkt_eval(rh.device_problem(lp), x.data_ptr(), y.data_ptr())
        assert rc == rh.OK
    assert rh.release_cached_memory() == 8 * (n + 8200)
    assert rh.release_cached_memory() == 0
