"""GPU: a frame may be let go of as soon as integrate has been called, and the
inputs of a fit as soon as it has been launched, although
the map's stream reads it later: its memory, device or pinned, is not given to
another tensor before."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

POSE = np.eye(4, dtype=np.float32)[:3].reshape(12)


@pytest.mark.parametrize("pinned", [False, True])
def test_a_frame_that_is_let_go_of_at_once(pinned):
    import torch
    from paper_2510_01592_gb300 import vm
    n = 200_000
    m = vm.VoxelMap((100, 100, 100), (0.0, 0.0, 0.0), 0.01)
    gen = torch.Generator().manual_seed(1)
    inside = torch.rand(n, 3, generator=gen) * 0.98 + 0.01
    busy = torch.rand(2_000_000, 3, generator=gen).cuda()

    def frame(points):
        if pinned:
            p = torch.empty(points.shape, pin_memory=True)
            p.copy_(points)
            return p
        return points.cuda()

    outside = torch.full((n, 3), 50.0)
    frame(outside)  # the allocator has a block of this size
    torch.cuda.synchronize()
    rounds = 12
    for _ in range(rounds):
        for _ in range(4):  # keeps the map's stream behind
            m.integrate(busy, POSE)
        m.integrate(frame(inside), POSE)
        later = frame(outside)  # takes the block if it is free
        del later
    torch.cuda.synchronize()
    s = m.stats()
    assert s["points_integrated"] + s["points_dropped"] == rounds * (n + 4 * len(busy))
    assert s["points_dropped"] == 0


def test_frames_without_a_segmentation_are_let_go_of():
    import gc
    import weakref

    import torch
    from paper_2510_01592_gb300 import vm
    m = vm.VoxelMap((40, 40, 40), (0.0, 0.0, 0.0), 0.01)
    kept = []
    for i in range(200):
        p = torch.rand(100, 3, device="cuda") * 0.4
        kept.append(weakref.ref(p))
        m.integrate(p, POSE)
        del p
    gc.collect()
    assert sum(r() is not None for r in kept) <= 64
    m.segment(vm.segment_params(min_cluster=1))
    gc.collect()
    assert not any(r() is not None for r in kept)


def test_a_launched_fit_holds_its_inputs_until_it_is_waited_for():
    import gc
    import weakref

    import torch
    from paper_2510_01592_gb300 import vm
    plan = vm.FitPlan(4, 4000, vm.segment_params(n_hyp=32))
    xyz, off = torch.rand(4000, 3, device="cuda"), torch.arange(0, 4001, 1000, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    refs = weakref.ref(xyz), weakref.ref(off)
    plan.launch(xyz, off)
    del xyz, off
    gc.collect()
    assert all(r() is not None for r in refs)
    plan.wait()
    gc.collect()
    assert not any(r() is not None for r in refs)
