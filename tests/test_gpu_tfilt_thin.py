"""The frame of a long, thin T image: its links take the whole grid, whichever
way the image lies, and the pairs are those of its transpose."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _flatten_us(f):
    from torch.profiler import ProfilerActivity, profile

    for _ in range(3):  # (the first session may see no kernels)
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            f()
            torch.cuda.synchronize()
        us = [e.device_time_total / e.count for e in p.key_averages() if "k_t_flatten" in e.key]
        if us and us[0] > 0:
            return us[0]
    pytest.skip("the profiler sees no kernels here")


def test_frame_rows_take_the_whole_grid():
    """2 rows of 2^21 against 2^21 rows of 3: before, a block per row took 3 ms
    for the former and 12 us for the latter."""
    import paper_2606_04801_gb300 as cp

    g = torch.Generator(device="cuda").manual_seed(4)
    wide = torch.rand((1, 1 << 21), generator=g, device="cuda")
    tall = wide.t().contiguous()
    a = _flatten_us(lambda: cp.persistence(wide, filtration="T"))
    b = _flatten_us(lambda: cp.persistence(tall, filtration="T"))
    assert a < 10 * b, (a, b)


@pytest.mark.parametrize("n", [1, 2, 255, 256, 257, 5000])
@pytest.mark.parametrize("rows", [1, 2, 3])
def test_thin_images_equal_their_transposes(n, rows):
    import paper_2606_04801_gb300 as cp

    g = torch.Generator(device="cuda").manual_seed(n)
    x = torch.randperm(rows * n, generator=g, device="cuda").float().view(rows, n)  # (no ties, whose order is by index)
    for y in (x.t().contiguous(), x.view(1, rows, n).permute(2, 1, 0).contiguous(), x.view(rows, 1, n).contiguous()):
        a, b = cp.persistence(x, filtration="T"), cp.persistence(y, filtration="T")
        top = 1 if y.dim() == 2 else 2
        key = lambda d, t: sorted(zip((d.dim == t).tolist(), d.birth.tolist(), d.death.tolist()))  # noqa: E731
        if y.dim() == 2:
            assert key(a, 1) == key(b, top)
        else:  # a sheet of voxels bounds no cavity; its components are the image's
            pa, pb = (sorted((u, v) for t, u, v in key(d, 0) if t) for d in (a, b))
            assert pa == pb
