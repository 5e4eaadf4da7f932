"""GPU: a map's segmentation takes the fit's kernels by the points its clusters
have, also when its first call could only go by the size of the scratch."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

POSE = np.array([1, 0, 0, 0, 0, 1, 0, 0, 0, 0, 1, 0], np.float32)


def _launches(vm, m, prm):
    a = vm.launch_count()
    m.segment(prm)
    return vm.launch_count() - a


def test_many_bricks_with_few_clustered_points():
    from paper_2510_01592_gb300 import vm
    rng = np.random.default_rng(1)
    prm = vm.segment_params(n_hyp=32)
    floor = (np.stack(np.meshgrid(np.arange(60), np.arange(60), [20]), -1).reshape(-1, 3) + 0.5) * 0.01
    want = None
    for spread in (0, 25000, 60000):  # scattered points: a brick each or so, none in a cluster
        m = vm.VoxelMap((800, 800, 100), (0.0, 0.0, 0.0), 0.01)
        pts = np.concatenate([floor, rng.uniform(0, 1, (spread, 3)) * [6.9, 7.9, 0.9] + [1.0, 0, 0]])
        m.integrate(pts.astype(np.float32), POSE)
        first = m.segment(prm)
        assert len(first["planes"]) >= 1
        m.segment(prm)
        n = _launches(vm, m, prm)
        captures = vm.capture_count()
        again = m.segment(prm)
        for key in ("planes", "hull_xy", "hull_xyz"):
            assert first[key].tobytes() == again[key].tobytes(), key
        m.reset()  # an emptied map keeps its kernels
        m.integrate(pts.astype(np.float32), POSE)
        assert _launches(vm, m, prm) == n and vm.capture_count() == captures
        if spread:
            assert m.stats()["bricks_allocated"] > 20000
        want = want or n
        assert n == want
