"""The 3D pruning pass at the edges of its 60 x 29 tiles, its plane chunks and
its code rows (widths that are and are not multiples of 4), against the
oracle: every field of every pair, with and without ties."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
FIELDS = ("birth", "death", "birth_cell", "death_cell", "birth_pixel", "death_pixel", "dim")


@pytest.fixture(scope="module")
def cp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2606_04801_gb300 as cp

    return cp


def _same(got, want, what):
    assert len(got) == len(want), f"{what}: {len(got)} pairs vs {len(want)}"
    for k in FIELDS:
        assert np.array_equal(got[k], want[k]), (what, k)


@pytest.mark.parametrize("shape", [(2, 29, 60), (3, 30, 61), (4, 28, 59), (5, 58, 120), (4, 59, 121), (2, 2, 181), (2, 88, 2),
                                   (64, 11, 40), (65, 12, 44), (130, 3, 5), (9, 31, 64), (7, 60, 65), (12, 40, 63)])
@pytest.mark.parametrize("kind", ["noise", "levels", "smooth", "plateau"])
def test_tile_edges(cp, shape, kind):
    rng = np.random.default_rng(sum(shape))
    img = {"noise": lambda: rng.random(shape, dtype=np.float32),
           "levels": lambda: rng.integers(0, 3, shape).astype(np.float32),
           "smooth": lambda: workloads.blurred(shape, 1.5, sum(shape)),
           "plateau": lambda: np.where(rng.random(shape) < 0.02, -1.0, 0.0).astype(np.float32)}[kind]()
    x = torch.from_numpy(img).cuda()
    _same(cp.persistence(x).numpy(), oracle.persistence(img), f"V {shape} {kind}")
    if kind != "smooth":
        _same(cp.persistence(x, filtration="T").numpy(), oracle.persistence_t(img), f"T {shape} {kind}")


def test_non_finite_at_tile_edges(cp):
    for at in [(0, 0, 0), (3, 28, 59), (3, 29, 60), (4, 30, 61), (2, 0, 60), (4, 30, 0)]:
        for v in (np.nan, np.inf, -np.inf):
            img = workloads.uniform((5, 31, 62), 1)
            img[at] = v
            with pytest.raises(cp.CpError) as e:
                cp.persistence(torch.from_numpy(img).cuda())
            assert e.value.code == -2
