"""GPU: a reset clears what was claimed and nothing less: a map that was filled,
scrolled, ray-cleared or driven past its pool holds, after a reset and a new
frame, what a new map holds after that frame."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

POSE = np.array([1, 0, 0, 0, 0, 1, 0, 0, 0, 0, 1, 0], np.float32)


@pytest.mark.parametrize("dims,capacity", [((8, 8, 8), 1), ((61, 47, 33), 0), ((61, 47, 33), 37), ((200, 9, 17), 0)])
def test_reset_equals_a_new_map(dims, capacity):
    from paper_2510_01592_gb300 import vm
    rng = np.random.default_rng(sum(dims) + capacity)
    ext = np.array(dims) * 0.05
    cloud = lambda n: (rng.uniform(0, 1, (n, 3)) * ext).astype(np.float32)
    used = vm.VoxelMap(dims, (0.0, 0.0, 0.0), 0.05, capacity)
    shift = np.array([1, 0, -1])
    used.integrate(cloud(6000), POSE)
    used.integrate(cloud(500), POSE, clear=True)
    used.scroll(shift)
    used.scroll(-shift)
    used.integrate(cloud(3000), POSE)
    for n in (0, 1, 700):
        used.reset()
        assert used.stats()["bricks_allocated"] == 0 and used.stats()["points_integrated"] == 0
        frame = cloud(n)
        if capacity:  # the pool's order of claims decides which bricks it holds: one brick's points only
            frame = np.minimum(frame, np.float32(0.39))
        new = vm.VoxelMap(dims, (0.0, 0.0, 0.0), 0.05, capacity)
        for m in (used, new):
            m.integrate(frame, POSE)
        a, b = used.stats(), new.stats()
        for k in ("points_integrated", "points_dropped", "points_no_capacity", "bricks_allocated", "status"):
            assert a[k] == b[k], k
        for x, y in zip(used.export_voxels(), new.export_voxels()):
            np.testing.assert_array_equal(x, y)
