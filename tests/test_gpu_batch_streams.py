"""A batch on the caller's stream: the stream destroyed before the batch, and calls that fail on it.
The failure is made on the host, by invalidating a stream capture, so that an asynchronous call on the
stream returns an error and the device stays as it is."""
import ctypes as C

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


@pytest.fixture(scope="module")
def cudart():
    try:
        return C.CDLL("libcudart.so")
    except OSError:
        return C.CDLL("/usr/local/cuda/lib64/libcudart.so")


def new_stream(cudart):
    st = C.c_void_p()
    assert cudart.cudaStreamCreateWithFlags(C.byref(st), 1) == 0
    return st


def run(b, rh, slot):
    while b.status(slot) == rh.STATUS_RUNNING:
        b.step(64)


def test_remove_reports_a_slot_it_could_not_clear(rh, cudart):
    lp = lpgen.make_standard_planted(seed=3, m=60, n=150)
    st = new_stream(cudart)
    with rh.Batch(1, 4 << 20, stream=st.value) as b:
        free0 = b.free_bytes()
        slot = b.add(lp, max_iters=64)
        run(b, rh, slot)
        graph = C.c_void_p()
        assert cudart.cudaStreamBeginCapture(st, 1) == 0
        assert cudart.cudaStreamSynchronize(st) != 0          # not allowed: the capture is invalid
        rc = rh.rhpdhg_batch_remove(b.b, slot)
        cudart.cudaStreamEndCapture(st, C.byref(graph))
        cudart.cudaGetLastError()
        assert rc != rh.OK
        assert b.poll(slot).iters == 64                       # the slot kept its result; now removed
        assert b.free_bytes() == free0
        slot = b.add(lp, max_iters=64)
        run(b, rh, slot)
        assert b.poll(slot).iters == 64
    assert cudart.cudaStreamDestroy(st) == 0


@pytest.mark.parametrize("last", ["step", "remove", "add"])
def test_batch_freed_after_its_stream(rh, cudart, last):
    """Work that add and remove leave on the stream is waited for, without the stream itself."""
    lp = lpgen.make_standard_planted(seed=3, m=60, n=150)
    st = new_stream(cudart)
    b = rh.Batch(2, 8 << 20, stream=st.value)
    slot = b.add(lp, max_iters=64)
    run(b, rh, slot)
    if last != "step":
        assert b.poll(slot).iters == 64
    if last == "add":
        b.add(lp, max_iters=64)
    assert cudart.cudaStreamDestroy(st) == 0
    b.close()
    with rh.Solver(lp, max_iters=64) as s:                    # the device still answers
        assert s.run().iters == 64
