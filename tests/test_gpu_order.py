"""The output order: every pair's place among the cells, through the bucket
sort, with output arrays and workspaces that are not 16- or 256-byte
aligned, few and many pairs per bucket, and outputs that are too small."""
import ctypes

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


def _call(lib, img, cap, out_off=0, ws_off=0):
    x = torch.from_numpy(img).cuda()
    nd = img.ndim
    dims = (ctypes.c_int64 * nd)(*img.shape)
    wsb = lib.cubical_persistence_workspace_size(nd, dims, 0)
    ws = torch.empty(wsb + ws_off, dtype=torch.uint8, device="cuda")
    out = torch.full((cap * 8 + 16 + out_off,), -7, dtype=torch.int32, device="cuda")
    cnt = ctypes.c_int64(0)
    fn = lib.cubical_persistence_2d if nd == 2 else lib.cubical_persistence_3d
    rc = fn(ctypes.c_void_p(x.data_ptr()), dims, ctypes.c_void_p(out.data_ptr() + 4 * out_off), cap, ctypes.byref(cnt),
            None, ctypes.c_void_p(ws.data_ptr() + ws_off), wsb, 0, None)
    o = out.cpu().numpy()
    assert (o[:out_off] == -7).all() and (o[out_off + 8 * cap :] == -7).all()  # nothing outside the output
    return rc, int(cnt.value), o[out_off : out_off + 8 * cap].reshape(cap, 8)


@pytest.mark.parametrize("img", [workloads.uniform((64, 65), 3), workloads.uniform((2, 2), 4),
                                 workloads.blurred((300, 410), 2.0, 5), workloads.uniform((24, 25, 26), 6),
                                 (np.indices((90, 91)).sum(0) % 2).astype(np.float32)],
                         ids=["noise2d", "tiny", "smooth2d", "noise3d", "checkerboard"])
@pytest.mark.parametrize("out_off,ws_off", [(0, 0), (1, 8), (2, 16), (3, 248)])
def test_unaligned_outputs_and_workspaces(cp, img, out_off, ws_off):
    lib = cp.load()
    want = oracle.persistence(img)
    rc, n, o = _call(lib, img, len(want), out_off, ws_off)
    assert rc == 0 and n == len(want)
    got = np.ascontiguousarray(o).view(cp.PAIR_DTYPE).reshape(-1)
    for k in ("birth", "death", "birth_cell", "death_cell", "birth_pixel", "death_pixel", "dim"):
        assert np.array_equal(got[k], want[k]), k


def test_short_output_holds_the_first_pairs(cp):
    img = workloads.uniform((50, 40), 7)
    want = oracle.persistence(img)
    rc, n, o = _call(cp.load(), img, 10)
    assert rc == -3 and n == len(want)
    assert np.array_equal(o[:, 2], want["birth_cell"][:10])
