"""Host time of a plan: it does not grow with the tuned bound on a task's planes
beyond the volumes' own depth."""
import ctypes
import time


def _plan_time(lib, shapes):
    k = len(shapes)
    ndims = (ctypes.c_int32 * k)(*[3] * k)
    dims = (ctypes.c_int64 * (3 * k))(*[v for s in shapes for v in s])
    best = float("inf")
    for _ in range(50):
        t0 = time.perf_counter()
        assert lib.cubical_persistence_batched_workspace_size(k, ndims, dims, 0) > 0
        best = min(best, time.perf_counter() - t0)
    return best


def test_plan_time_follows_the_volumes():
    from paper_2606_04801_gb300 import _lib, build

    build.build()
    lib = _lib.load()
    saved = lib.cp_get_tuning(1)
    try:
        times = {}
        for zc in (16, 4096):
            assert lib.cp_set_tuning(1, zc) == 0
            times[zc] = _plan_time(lib, [(16, 20, 30)] * 128)
        # the same candidates are looked at (before: 256 times as many)
        assert times[4096] < 10 * times[16], times
    finally:
        assert lib.cp_set_tuning(1, saved) == 0
