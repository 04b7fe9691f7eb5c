"""A batched slot's result by every way it leaves the device: into host memory, into device memory,
and polled twice, with the certificate of an infeasible LP, an LP without rows, and slots in FP64 and
mixed precision.  The ways hand out the same numbers, so they are compared bit for bit."""
import numpy as np
import pytest

from paper_2407_16144_gb300 import lpgen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rh():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2407_16144_gb300 import _build, rhpdhg
    _build.build()
    rhpdhg.load()
    return rhpdhg


LPS = {
    "planted": lambda: lpgen.make_standard_planted(seed=3, m=130, n=321),
    "infeasible": lambda: lpgen.make_primal_infeasible(5, 150, 300),
    "unbounded": lambda: lpgen.make_dual_infeasible(5, 150, 300),
    "no_rows": lambda: lpgen.make_box_lp(1, n=20),
}


def device_poll(rh, b, slot, n, m):
    import torch
    v = [torch.full((k,), -1.0, dtype=torch.float64, device="cuda") for k in (n, m, n, m)]
    r = rh.rhpdhg_result()
    r.out_memory = rh.MEM_DEVICE
    r.x, r.y, r.cert_x, r.cert_y = (t.data_ptr() if t.numel() else None for t in v)
    assert rh.rhpdhg_batch_poll(b.b, slot, r) == rh.OK
    return r, [t.cpu().numpy() for t in v]


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("name", list(LPS))
def test_device_poll_equals_host_poll(rh, name, prec):
    lp = LPS[name]()
    with rh.Batch(4, 64 << 20) as b:
        other = b.add(lpgen.make_standard_planted(seed=4, m=60, n=150), max_iters=64)
        s = b.add(lp, precision=prec, eps_rel_kkt=1e-6, max_iters=20_000)
        while b.status(s) == rh.STATUS_RUNNING or b.status(other) == rh.STATUS_RUNNING:
            b.step(64)
        first = b.poll(s, remove=False)
        r, vecs = device_poll(rh, b, s, lp.n, lp.m)
        b.step(64)                                 # a finished slot stays as it is
        again = b.poll(s, remove=False)
    if name == "infeasible":
        assert first.status == rh.STATUS_PRIMAL_INFEASIBLE
    for host in (first, again):
        for k in ("status", "iters", "restarts", "cert_source", "primal_obj", "dual_obj", "eta",
                  "omega", "sigma_max", "rel_p", "rel_d", "rel_gap"):
            assert np.array_equal(getattr(host, k), getattr(r, k), equal_nan=True), k
        for want, got in zip((host.x, host.y, host.cert_x, host.cert_y), vecs):
            assert np.array_equal(want, got)


def test_batch_keeps_no_device_memory_outside_its_arena(rh):
    lp = lpgen.make_standard_planted(seed=3, m=130, n=321)
    rh.release_cached_memory()
    with rh.Batch(2, 16 << 20) as b:
        s = b.add(lp, max_iters=64)
        while b.status(s) == rh.STATUS_RUNNING:
            b.step(64)
        device_poll(rh, b, s, lp.n, lp.m)
        b.poll(s)
    assert rh.release_cached_memory() == 0
