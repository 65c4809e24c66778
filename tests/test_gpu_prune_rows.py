"""The 2D pruning pass at the edges of its 30 x 30 tiles, with one to eight
warps per tile, alone and batched, against the oracle: every field of every
pair."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
FIELDS = ("birth", "death", "birth_cell", "death_cell", "birth_pixel", "death_pixel", "dim")


def _image(shape, kind):
    rng = np.random.default_rng(sum(shape))
    return {"noise": lambda: rng.random(shape, dtype=np.float32),
            "levels": lambda: rng.integers(0, 3, shape).astype(np.float32),
            "plateau": lambda: np.where(rng.random(shape) < 0.02, -1.0, 0.0).astype(np.float32)}[kind]()


def _same(got, want, what):
    assert len(got) == len(want), f"{what}: {len(got)} pairs vs {len(want)}"
    for k in FIELDS:
        assert np.array_equal(got[k], want[k]), (what, k)


@pytest.mark.parametrize("shape", [(2, 2), (3, 32), (4, 31), (5, 62), (6, 30), (9, 63), (13, 1000), (3001, 7), (640, 962), (1301, 517),
                                   (47, 12007), (30, 30), (31, 60), (61, 91), (500, 600), (1500, 1501)])
@pytest.mark.parametrize("kind", ["noise", "levels", "plateau"])
def test_task_edges(shape, kind):
    import paper_2606_04801_gb300 as cp

    img = _image(shape, kind)
    x = torch.from_numpy(img).cuda()
    _same(cp.persistence(x).numpy(), oracle.persistence(img), f"V {shape} {kind}")
    if shape[0] < 64:
        _same(cp.persistence(x, filtration="T").numpy(), oracle.persistence_t(img), f"T {shape} {kind}")


def test_batch_of_uneven_images():
    import paper_2606_04801_gb300 as cp

    imgs = [_image(s, "levels") for s in [(5, 31), (700, 901), (2, 63), (129, 33)]] + [workloads.uniform((3, 4, 5), 2)]
    got = cp.persistence_batched([torch.from_numpy(v).cuda() for v in imgs]).numpy()
    for i, v in enumerate(imgs):
        _same(got[got["item"] == i], oracle.persistence(v), str(v.shape))
