"""The output launch with fewer thread blocks than the chunks of its buckets (a
device or a partition with few SMs): the same pairs in the same order."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("blocks", [1, 2, 7, 63, 127, 128, 10 ** 6])
@pytest.mark.parametrize("shape", [(2, 2), (300, 17), (1000, 700), (30, 40, 50), (90, 100, 110)])
def test_few_blocks(shape, blocks):
    import paper_2606_04801_gb300 as cp

    lib = cp.load()
    g = torch.Generator(device="cuda").manual_seed(9)
    x = torch.randint(0, 40, shape, generator=g, device="cuda").float()
    want = cp.persistence(x).raw
    dims = (ctypes.c_int64 * len(shape))(*shape)
    ws_bytes = lib.cubical_persistence_workspace_size(len(shape), dims, 0)
    ws = torch.full((ws_bytes,), 0xA5, dtype=torch.uint8, device="cuda")
    out = torch.empty((x.numel() + 1, 8), dtype=torch.int32, device="cuda")
    cnt = ctypes.c_int64(0)
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    rc = lib.cubical_persistence_debug_order_blocks(len(shape), p(x), dims, p(out), out.shape[0], ctypes.byref(cnt), None, p(ws),
                                                    ws_bytes, blocks, None)
    assert rc == 0 and torch.equal(out[: cnt.value], want)
