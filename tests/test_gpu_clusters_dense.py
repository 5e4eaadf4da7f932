"""GPU: clustering where its pieces change over, against the oracle bit for bit:
bricks with every voxel occupied (their records do not fit the staging area),
tens of thousands of components (beyond what one SM joins), thousands of
one-voxel clusters (more than the first scratch holds, and than the placement
counts in shared memory), every voxel in one cluster, the far corner of a 16 m
map, a scrolled window of odd size."""
import numpy as np
import pytest

from parity import compare_labels, compare_planes

pytestmark = pytest.mark.gpu

POSE = np.array([1, 0, 0, 0, 0, 1, 0, 0, 0, 0, 1, 0], np.float32)


@pytest.mark.parametrize("dims,density,shift,kw", [
    ((24, 16, 16), 1.0, (0, 0, 0), dict(classify=0, d_th=0.2, theta_ccl_deg=179.0, min_cluster=1)),
    ((24, 16, 16), 1.0, (0, 0, 0), dict(classify=0, d_th=0.04, theta_ccl_deg=40.0, min_cluster=2)),
    ((40, 33, 29), 0.35, (0, 0, 0), dict(classify=0, theta_ccl_deg=20.0, min_cluster=1)),
    ((96, 96, 64), 0.4, (0, 0, 0), dict(classify=0, d_th=0.06, theta_ccl_deg=6.0, min_cluster=6)),
    ((319, 319, 319), 0.1, (0, 0, 0), dict(classify=1, theta_step_deg=50.0, theta_ccl_deg=60.0, min_cluster=5)),
    ((45, 27, 51), 0.5, (2, -1, 3), dict(classify=1, theta_step_deg=50.0, theta_ccl_deg=60.0, min_cluster=5)),
])
def test_dense_clusters(orc, dims, density, shift, kw):
    from paper_2510_01592_gb300 import vm
    rng = np.random.default_rng(int(1000 * density) + dims[0])
    gm, om = vm.VoxelMap(dims, (0.0, 0.0, 0.0), 0.05), orc.OracleMap(dims, (0.0, 0.0, 0.0), 0.05)
    if any(shift):
        gm.scroll(np.array(shift))
        om.scroll(np.array(shift))
    # of a large map the far corner only: the largest coordinates a map can have
    cell = np.stack(np.meshgrid(*[np.arange(max(0, d - 96), d) for d in dims], indexing="ij"), -1).reshape(-1, 3)
    cell = cell[rng.uniform(0, 1, len(cell)) < density] + 8 * np.array(shift)
    pts = ((cell + rng.uniform(0.1, 0.9, cell.shape)) * 0.05).astype(np.float32)
    gm.integrate(pts, POSE)
    om.integrate(pts, POSE)
    ores = om.segment(orc.make_params(n_hyp=8, **kw))
    for _ in range(2):  # the second time with the scratch that the first one grew
        gres = gm.segment(vm.segment_params(n_hyp=8, **kw))
        compare_labels(gm.export_labels(), ores["voxels"])
        compare_planes(gres, ores, gm.export_clusters(), check_refit=False)
