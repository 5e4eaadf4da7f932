"""GPU: maps of noise, with far more components and clusters than surfaces give.
Their numbering and placement (several CTAs, fewer warps with counts of their
own, tile by tile) against the oracle bit for bit, and that these stages do not
outgrow the others."""
import numpy as np
import pytest

from parity import compare_labels, compare_planes

pytestmark = pytest.mark.gpu

POSE = np.array([1, 0, 0, 0, 0, 1, 0, 0, 0, 0, 1, 0], np.float32)


def _noise(dims, density, seed, surfaces=False):
    """Points in random cells; surfaces: also a floor and a wall, clusters that every tile has a part of."""
    rng = np.random.default_rng(seed)
    cell = np.stack(np.meshgrid(*[np.arange(d) for d in dims], indexing="ij"), -1).reshape(-1, 3)
    keep = rng.uniform(0, 1, len(cell)) < density
    at = rng.uniform(0.1, 0.9, cell.shape)
    if surfaces:
        for axis, where in ((2, 11), (0, 37)):
            on = cell[:, axis] == where
            keep = np.where(on, True, keep & (np.abs(cell[:, axis] - where) > 3))
            at[on, axis] = 0.5
    return ((cell + at)[keep] * 0.01).astype(np.float32)


@pytest.mark.parametrize("dims,density,surfaces,kw", [
    ((96, 96, 64), 0.10, False, dict(d_th=0.012, min_cluster=3)),     # hundreds of clusters, tens of thousands of components
    ((160, 160, 80), 0.10, False, dict(d_th=0.012, min_cluster=2)),   # thousands: a warp or a few count in each CTA
    ((160, 160, 80), 0.05, False, dict(d_th=0.05, min_cluster=1)),    # tens of thousands: tile by tile
    ((160, 160, 80), 0.05, True, dict(d_th=0.05, min_cluster=1)),     # and two clusters through every tile
    ((160, 160, 80), 0.05, True, dict(d_th=0.05, min_cluster=100)),   # of which nothing but those is kept
])
def test_many_components_and_clusters(orc, dims, density, surfaces, kw):
    from paper_2510_01592_gb300 import vm
    gm, om = vm.VoxelMap(dims, (0.0, 0.0, 0.0), 0.01), orc.OracleMap(dims, (0.0, 0.0, 0.0), 0.01)
    pts = _noise(dims, density, dims[0] + surfaces, surfaces)
    gm.integrate(pts, POSE)
    om.integrate(pts, POSE)
    ores = om.segment(orc.make_params(n_hyp=4, classify=0, **kw))
    for _ in range(2):  # the second time with the scratch that the first one grew
        gres = gm.segment(vm.segment_params(n_hyp=4, classify=0, **kw))
        compare_labels(gm.export_labels(), ores["voxels"])
        compare_planes(gres, ores, gm.export_clusters(), check_refit=False)


@pytest.mark.parametrize("density,min_cluster", [(0.05, 1), (0.4, 50)])
def test_clusters_of_noise_cost_no_more_than_its_voxels(density, min_cluster):
    """The numbering, the placement and the lists of 100 thousand clusters, or of a million components without one, take
    at most three times as long as the means and normals of the same voxels."""
    from paper_2510_01592_gb300 import vm
    m = vm.VoxelMap((200, 200, 100), (0.0, 0.0, 0.0), 0.01, stage_timing=True)
    m.integrate(_noise((200, 200, 100), density, 3), POSE)
    prm = vm.segment_params(n_hyp=4, classify=0, min_cluster=min_cluster)
    for _ in range(3):
        m.segment(prm)
    m.stage_times()
    best = None
    for _ in range(5):
        m.segment(prm)
        t = {k: v[0] for k, v in m.stage_times().items()}
        ratio = t["clusters"] / (t["finalize"] + t["moments"] + t["eigen"])
        best = ratio if best is None else min(best, ratio)
    assert best < 3.0, best


def test_the_first_segmentation_of_noise_is_not_held_up():
    """A map's first segmentation goes by no counts, and is repeated where the scratch has no room for the clusters: both
    runs' clustering together take at most ten times as long as the means and normals."""
    from paper_2510_01592_gb300 import vm
    best = None
    for _ in range(3):
        m = vm.VoxelMap((200, 200, 100), (0.0, 0.0, 0.0), 0.01, stage_timing=True)
        m.integrate(_noise((200, 200, 100), 0.05, 3), POSE)
        m.stage_times()
        m.segment(vm.segment_params(n_hyp=4, classify=0, min_cluster=1))
        t = {k: v[0] for k, v in m.stage_times().items()}
        ratio = t["clusters"] / (t["finalize"] + t["moments"] + t["eigen"])
        best = ratio if best is None else min(best, ratio)
        m.close()
    assert best < 10.0, best
