"""Long straight descents of a 2D image in each direction: the links of the
pruning pass are the restatement's, the pairs the oracle's, and the walks take
them several pixels at a time."""
import ctypes

import numpy as np
import pytest

import oracle
from prune_restatement import Pruned
from test_gpu_stages import _check

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
FIELDS = ("birth", "death", "birth_cell", "death_cell", "birth_pixel", "death_pixel", "dim")


@pytest.fixture(scope="module")
def cp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2606_04801_gb300 as cp

    return cp


def _valleys(shape, axis, sign, seed, ties=False):
    """Straight valleys that fall towards one end of an axis, with noise that
    stays below the slope; ties: in whole numbers, two pixels to a step."""
    rng = np.random.default_rng(seed)
    along, across = np.indices(shape)[axis].astype(np.float64), np.indices(shape)[1 - axis]
    x = sign * along + 50 * np.sin(across * (2 * np.pi / 8)) + 0.5 * rng.random(shape)
    return np.floor(x / 2 if ties else x * 64).astype(np.float32)


@pytest.mark.parametrize("shape", [(24, 130), (130, 24), (61, 93), (2, 67), (67, 2), (31, 30)])
@pytest.mark.parametrize("ties", [False, True])
@pytest.mark.parametrize("axis,sign", [(0, 1), (0, -1), (1, 1), (1, -1)])
def test_links_and_pairs(cp, shape, ties, axis, sign):
    for seed, up in ((1, 1), (2, -1)):  # valleys, and ridges for the dual's links
        img = up * _valleys(shape, axis, sign, seed, ties)
        _check(cp, cp.load(), img)
        x = torch.from_numpy(img).cuda()
        for filt, want in (("V", oracle.persistence(img)), ("T", oracle.persistence_t(img))):
            got = cp.persistence(x, filtration=filt).numpy()
            assert len(got) == len(want)
            for k in FIELDS:
                assert np.array_equal(got[k], want[k]), (filt, k)


def _depth(par):
    p = np.asarray(par, dtype=np.int64)
    d = (p != np.arange(len(p))).astype(np.int64)
    while not np.array_equal(p, p[p]):
        d, p = d + d[p], p[p]
    return d


@pytest.mark.parametrize("axis,sign", [(0, 1), (0, -1), (1, 1), (1, -1)])
def test_walks_take_several_pixels_at_a_time(cp, axis, sign):
    """A straight run through a tile (30 pixels) is 9 steps at most (7 of four, 2
    of one), and a path has a few more at its ends and bends: at most 0.45 of the
    pixels and 8 per survivor, of both lists (up and +y: fewer)."""
    lib = cp.load()
    shape = (24, 600) if axis else (600, 24)
    for up in (1, -1):
        img = up * _valleys(shape, axis, sign, 3)
        H, W = shape
        ref = Pruned(lib, img)
        d0, dt = _depth(ref.par0), _depth(ref.part)
        pixels = [0, 0]
        for dual, keys in enumerate((ref.s0_keys(), ref.st_keys())):
            for k in keys:
                v, n = (k >> 5) & (1 << 27) - 1, (k & 31) >> 1
                y, x, dy, dx = v // W, v % W, n // 3 - 1, n % 3 - 1
                if not dual:
                    ends = [d0[v], d0[v + dy * W + dx]]
                else:  # the top cells on the facet's two sides
                    ends = []
                    for s in (-1, 0):
                        cy, cx = (y + s if dy == 0 else y - (dy < 0)), (x + s if dx == 0 else x - (dx < 0))
                        ends.append(dt[cy * (W - 1) + cx] if 0 <= cy < H - 1 and 0 <= cx < W - 1 else 0)
                pixels[dual] += max(ends)
        n = [len(ref.s0_keys()), len(ref.st_keys())]
        dims = (ctypes.c_int64 * 2)(*shape)
        ws_bytes = lib.cubical_persistence_workspace_size(2, dims, 0)
        ws = torch.empty(ws_bytes, dtype=torch.uint8, device="cuda")
        out = torch.empty((img.size, 8), dtype=torch.int32, device="cuda")
        t = torch.from_numpy(img).cuda()
        cnt = ctypes.c_int64(0)
        p = lambda a: ctypes.c_void_p(a.data_ptr())  # noqa: E731
        assert lib.cubical_persistence_2d(p(t), dims, p(out), img.size, ctypes.byref(cnt), None, p(ws), ws_bytes, 0, None) == 0
        act, us, hops = (ctypes.c_uint32 * 48)(), (ctypes.c_double * 48)(), (ctypes.c_uint64 * 48)()
        assert max(pixels) > 50 * max(n)  # (there are long paths)
        for dual in (0, 1):
            assert lib.cubical_persistence_uf_trace2(p(ws), dual, act, us, None, hops, 48, None) == 2 and act[0] == n[dual]
            assert hops[0] <= 0.45 * pixels[dual] + 8 * n[dual], (up, dual, hops[0], pixels[dual], n[dual])
