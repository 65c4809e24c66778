"""The H1 time budget covers the rewriting of the columns and the rounds
together, and a spent one stops the rounds alone."""
import ctypes
import math

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def cp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2606_04801_gb300 as cp

    return cp


def _full(lib, xs):
    """One batched call with everything sized; its code, pairs and H1 information."""
    k = len(xs)
    ptrs = (ctypes.c_void_p * k)(*[x.data_ptr() for x in xs])
    ndims = (ctypes.c_int32 * k)(*[3] * k)
    dims = (ctypes.c_int64 * (3 * k))(*[v for x in xs for v in x.shape])
    n = sum(x.numel() for x in xs)
    ms, pool = 2 * n + 65536, 60 * n + 65536
    ws_bytes = lib.cubical_persistence_full_batched_workspace_size(k, ndims, dims, ms, pool)
    ws = torch.empty(ws_bytes, dtype=torch.uint8, device="cuda")
    out = torch.empty((3 * n, 8), dtype=torch.int32, device="cuda")
    cnt = ctypes.c_int64(0)
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    rc = lib.cubical_persistence_full_batched(k, ptrs, ndims, dims, p(out), out.shape[0], ctypes.byref(cnt), None, p(ws), ws_bytes,
                                              ms, pool, None)
    info = (ctypes.c_int64 * 13)()
    assert lib.cubical_persistence_full_info(p(ws), k, ndims, dims, ms, pool, info, 13, None) == 0
    return rc, out[: cnt.value], list(info)


def test_one_budget_for_both(cp):
    """1.2 times the rounds' own time is less than both take (32 volumes of 64^3
    noise: 7.2 ms and 13.4 ms), so the call stops; 4 times is enough."""
    lib = cp.load()
    g = torch.Generator(device="cuda").manual_seed(1)
    xs = [torch.rand((64, 64, 64), generator=g, device="cuda") for _ in range(32)]
    old = lib.cp_get_tuning(4)
    for _ in range(2):
        rc, want, info = _full(lib, xs)
        assert rc == 0
    rounds_ms = (info[11] + info[12]) / 1e6
    try:
        assert lib.cp_set_tuning(4, math.ceil(1.2 * rounds_ms)) == 0
        assert _full(lib, xs)[0] == -5  # CP_ERR_TIMEOUT
        assert lib.cp_set_tuning(4, math.ceil(4 * rounds_ms)) == 0
        rc, got, _ = _full(lib, xs)
        assert rc == 0 and torch.equal(got, want)
    finally:
        assert lib.cp_set_tuning(4, old) == 0


def test_a_budget_of_zero_stops_after_the_first_round(cp):
    """Small volumes whose columns that left their stars need no addition to one
    another are done in that round, and the call succeeds."""
    lib = cp.load()
    g = torch.Generator(device="cuda").manual_seed(2)
    xs = [torch.rand((3, 4, 3), generator=g, device="cuda") for _ in range(100)]
    want = [_full(lib, [x]) for x in xs]
    old = lib.cp_get_tuning(4)
    try:
        assert lib.cp_set_tuning(4, 0) == 0
        got = [_full(lib, [x]) for x in xs]
    finally:
        assert lib.cp_set_tuning(4, old) == 0
    assert all(rc == 0 for rc, _, _ in want)
    done = 0
    for (_, pairs, _), (rc, mine, info) in zip(want, got):
        assert rc in (0, -5)
        if rc == 0:
            assert torch.equal(mine, pairs)
            done += info[9] > 0
    assert done > 0  # of those with columns that left their stars
