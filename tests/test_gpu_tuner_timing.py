"""What the autotuner times as the pruning pass is that pass: the call's start
and one kernel per kind of item, and nothing that the calls do not run."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("shapes,kernels", [([(64, 48, 40)], 1), ([(64, 48)], 1), ([(64, 48), (16, 20, 30)], 2)])
def test_the_tuner_times_the_pruning_pass_alone(shapes, kernels):
    import paper_2606_04801_gb300 as cp
    from paper_2606_04801_gb300 import autotune

    lib = cp.load()
    xs = [torch.rand(s, device="cuda") for s in shapes]
    before = lib.cp_launch_count()
    assert autotune._time_prune(xs, 3) > 0
    assert lib.cp_launch_count() - before == 4 * (1 + kernels)
    # and what it ran leaves the context and the library as they were
    assert len(cp.persistence_batched(xs)) > 0
