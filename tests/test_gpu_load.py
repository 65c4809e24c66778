"""BatchedPersistence.load: the packed inputs hold every item's values, from
sources and to places on every 16-byte phase, and from the tensors that take
the general copy (host, other types, strided, parts of the batch itself)."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SHAPES = [(2, 2), (3, 5), (64, 64), (33, 31, 4), (4096, 2), (4095, 3), (2, 2, 3), (61, 67), (16, 16, 16), (129, 257)]


def _at(phase, shape, dev="cuda"):
    n = 1
    for v in shape:
        n *= v
    return torch.rand(n + 4, device=dev)[phase : phase + n].view(shape)


@pytest.mark.parametrize("phase", [0, 1, 2, 3])
def test_every_phase(phase):
    import paper_2606_04801_gb300 as cp

    bp = cp.BatchedPersistence(SHAPES)
    for turn in range(2):
        xs = [_at((phase + turn * i) % 4, s) for i, s in enumerate(SHAPES)]
        bp.load(xs)
        assert torch.equal(bp.x, torch.cat([v.reshape(-1) for v in xs]))


def test_general_copies_and_refusals():
    import paper_2606_04801_gb300 as cp

    shapes = [(5, 6)] * 10
    bp = cp.BatchedPersistence(shapes)
    xs = [torch.rand(5, 6), torch.rand(5, 6).numpy(), torch.rand(5, 6).double().cuda(), torch.rand(6, 5).cuda().t(),
          torch.rand(30).cuda(), torch.rand(1, 5, 6).cuda(), torch.rand(5, 6).tolist(), torch._neg_view(torch.rand(5, 6).cuda()),
          torch.randint(0, 9, (5, 6)).cuda(), torch.rand(5, 6).cuda()]
    bp.load(xs)
    assert torch.equal(bp.x, torch.cat([torch.as_tensor(v).to("cuda", torch.float32).reshape(-1) for v in xs]))
    before = bp.views[1].clone()
    bp.load([bp.views[1]] + [bp.views[0]] + xs[2:])  # in order, as copies one after the other
    assert torch.equal(bp.views[0], before) and torch.equal(bp.views[1], before)
    with pytest.raises(RuntimeError):
        bp.load(xs[:-1] + [torch.rand(5, 7).cuda()])
    with pytest.raises(ValueError):
        bp.load(xs[:-1])


def test_items_of_the_batch_as_sources_in_list_order():
    """A source that is a part of the batch sees the items before it in the
    list loaded and those after it not, whatever way each is copied."""
    import paper_2606_04801_gb300 as cp

    bp = cp.BatchedPersistence([(5, 6)] * 6)
    old = [torch.rand(5, 6).cuda() for _ in range(6)]
    bp.load(old)
    new = [torch.rand(5, 6).cuda() for _ in range(6)]
    src = [new[0], bp.views[0], bp.views[3], new[3], bp.views[3].double(), bp.views[2].t().contiguous().t()]
    want = [new[0], new[0], old[3], new[3], old[3], old[2]]  # (the last two are copies made before the call)
    bp.load(src)
    for i, v in enumerate(want):
        assert torch.equal(bp.views[i], v), i
    bp.load([new[1], bp.views[0].view(6, 5).t(), new[2], new[3], new[4], new[5]])  # strided
    assert torch.equal(bp.views[1], new[1].view(6, 5).t())


def test_device_without_index_takes_one_launch():
    import paper_2606_04801_gb300 as cp

    lib = cp.load()
    for device in (None, "cuda", "cuda:0"):
        bp = cp.BatchedPersistence([(5, 6)] * 4, device=device)
        xs = [torch.rand(5, 6).cuda() for _ in range(4)]
        before = lib.cp_launch_count()
        bp.load(xs)
        assert lib.cp_launch_count() - before == 1, device
        assert torch.equal(bp.x, torch.cat([v.reshape(-1) for v in xs]))


def test_autograd_sees_a_load_as_it_sees_a_copy():
    """A value saved for backward that a load overwrites is an error, not a
    gradient of the new values; tangents of forward mode are copied; a batch
    made in inference mode takes loads there alone."""
    import torch.autograd.forward_ad as fw

    import paper_2606_04801_gb300 as cp

    def one():
        return torch.rand(5, 6).cuda()

    bp = cp.BatchedPersistence([(5, 6)] * 2)
    bp.load([one(), one()])
    w = torch.rand(5, 6, device="cuda", requires_grad=True)
    y = (bp.views[1] * w).sum()
    bp.load([one(), one()])
    with pytest.raises(RuntimeError, match="modified by an inplace operation"):
        y.backward()
    with fw.dual_level():
        t = torch.rand(5, 6).cuda()
        bp.load([fw.make_dual(one(), t), one()])
        assert torch.equal(fw.unpack_dual(bp.views[0]).tangent, t)
    with torch.inference_mode():
        bi = cp.BatchedPersistence([(5, 6)] * 2)
        xs = [one(), one()]
        bi.load(xs)
        assert torch.equal(bi.x, torch.cat([v.reshape(-1) for v in xs]))
    with pytest.raises(RuntimeError):
        bi.load([one(), one()])


def test_a_tensor_without_memory_is_zeros():
    import paper_2606_04801_gb300 as cp

    bp = cp.BatchedPersistence([(5, 6)] * 2)
    xs = [torch.rand(5, 6).cuda() for _ in range(2)]
    bp.load(xs)
    bp.load([torch._efficientzerotensor((5, 6), device="cuda"), xs[1]])
    assert not bp.views[0].any() and torch.equal(bp.views[1], xs[1])
