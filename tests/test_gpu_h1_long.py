"""Whole diagrams of volumes whose loops bound large discs: the columns that
leave their star outgrow the first launch's shared memory, then the second's
(they go on in the column pool), then the part of the pool it may use."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
FIELDS = ("birth", "death", "birth_cell", "death_cell", "birth_pixel", "death_pixel", "dim")


@pytest.mark.parametrize("side,pool", [(40, 0), (150, 0), (260, 0), (260, 2000)])
def test_long_loops(side, pool):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2606_04801_gb300 as cp

    rng = np.random.default_rng(side)
    c = (side - 1) / 2
    y, x = np.mgrid[:side, :side]
    ring = np.abs(np.hypot(y - c, x - c) - 0.85 * c)  # a valley along a circle, a peak in its middle
    img = (ring[None] + 0.01 * rng.random((3, side, side))).astype(np.float32)
    got = cp.persistence_full(torch.from_numpy(img).cuda(), pool_entries=pool).numpy()
    want = oracle.persistence_full(img)
    assert len(got) == len(want)
    for k in FIELDS:
        assert np.array_equal(got[k], want[k]), k
    loops = got[got["dim"] == 1]
    assert (loops["death"] - loops["birth"]).max() > 0.8 * 0.85 * c  # the circle's loop
