"""Failure detection without a GPU fault: bad arguments and non-finite
input are reported as error codes (see test_gpu_parity.py); a bounded device
wait that nothing satisfies gives up after its limit, reports
CP_ERR_TIMEOUT, and leaves the context usable."""
import ctypes
import time

import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def cp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2606_04801_gb300 as cp

    return cp


def test_bounded_wait_gives_up(cp):
    lib = cp.load()
    ws = torch.zeros(8192, dtype=torch.uint8, device="cuda")
    t0 = time.perf_counter()
    rc = lib.cubical_persistence_debug_wait_timeout(ctypes.c_void_p(ws.data_ptr()), ws.numel(), 50_000, None)
    dt = time.perf_counter() - t0
    assert rc == -5  # CP_ERR_TIMEOUT
    assert dt < 5.0
    # the context is still usable afterwards
    img = workloads.uniform((40, 30), 5)
    got = cp.persistence(torch.from_numpy(img).cuda()).numpy()
    want = oracle.persistence(img)
    assert np.array_equal(got["birth_cell"], want["birth_cell"])
    assert lib.cubical_persistence_debug_wait_timeout(ctypes.c_void_p(ws.data_ptr()), 100, 50_000, None) == -1


@pytest.mark.parametrize("shape", [(40, 30), (700, 500), (20, 30, 40)])
def test_output_barrier_gives_up(cp, shape):
    """A grid barrier of the output launch that is never reached: every block
    leaves, the call fails, nothing is reported or written, and the same
    workspace serves the next call."""
    lib = cp.load()
    img = workloads.uniform(shape, 5)
    x = torch.from_numpy(img).cuda()
    dims = (ctypes.c_int64 * len(shape))(*shape)
    ws_bytes = lib.cubical_persistence_workspace_size(len(shape), dims, 0)
    ws = torch.full((ws_bytes,), 0xA5, dtype=torch.uint8, device="cuda")  # nothing in it is a valid index
    out = torch.full((img.size, 8), -7, dtype=torch.int32, device="cuda")
    d_count = torch.full((1,), 77, dtype=torch.int64, device="cuda")
    cnt = ctypes.c_int64(77)
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    rc = lib.cubical_persistence_debug_order_timeout(len(shape), p(x), dims, p(out), img.size, ctypes.byref(cnt), p(d_count),
                                                     p(ws), ws_bytes, 20_000, None)
    assert rc == -5  # CP_ERR_TIMEOUT
    assert cnt.value == 0 and int(d_count) == 0 and bool((out == -7).all())
    fn = lib.cubical_persistence_2d if len(shape) == 2 else lib.cubical_persistence_3d
    rc = fn(p(x), dims, p(out), img.size, ctypes.byref(cnt), p(d_count), p(ws), ws_bytes, 0, None)
    assert rc == 0 and int(d_count) == cnt.value
    want = cp.persistence(x).raw
    assert torch.equal(out[: cnt.value], want)
    bad = lib.cubical_persistence_debug_order_timeout
    assert bad(len(shape), p(x), dims, p(out), img.size, ctypes.byref(cnt), None, p(ws), ws_bytes, 0, None) == -1
    assert bad(len(shape), p(x), dims, p(out), img.size, ctypes.byref(cnt), None, p(ws), 100, 10, None) == -1


def test_nonfinite_volume_fails_cleanly(cp):
    vol = workloads.blurred((20, 30, 40), 2.0, 6)
    vol[7, 11, 13] = np.nan
    with pytest.raises(cp.CpError) as e:
        cp.persistence(torch.from_numpy(vol).cuda())
    assert e.value.code == -2
    vol[7, 11, 13] = np.inf
    with pytest.raises(cp.CpError) as e:
        cp.persistence(torch.from_numpy(vol).cuda())
    assert e.value.code == -2
    vol[7, 11, 13] = 0.5  # and a clean call afterwards
    got = cp.persistence(torch.from_numpy(vol).cuda()).numpy()
    assert len(got) == len(oracle.persistence(vol))
