"""GPU: clustering when the list of joined component pairs has no room for all of
them: the pairs beyond join a forest of their own, which is merged with the
listed ones.  Labels, cluster points and planes against the oracle, with room for
no pair, one, and some."""
import numpy as np
import pytest

from parity import compare_labels, compare_planes

pytestmark = pytest.mark.gpu

POSE = np.array([1, 0, 0, 0, 0, 1, 0, 0, 0, 0, 1, 0], np.float32)


@pytest.mark.parametrize("cap", [0, 1, 300])
@pytest.mark.parametrize("dims,density,kw", [
    ((40, 33, 29), 0.35, dict(theta_ccl_deg=20.0, min_cluster=1)),                # a few thousand components
    ((96, 96, 64), 0.4, dict(d_th=0.06, theta_ccl_deg=6.0, min_cluster=6)),       # more than one SM joins
    ((64, 64, 24), 0.9, dict(d_th=0.2, theta_ccl_deg=179.0, min_cluster=1)),      # one cluster
])
def test_pairs_beyond_the_list(orc, monkeypatch, cap, dims, density, kw):
    from paper_2510_01592_gb300 import vm
    rng = np.random.default_rng(dims[0])
    cell = np.stack(np.meshgrid(*[np.arange(d) for d in dims], indexing="ij"), -1).reshape(-1, 3)
    cell = cell[rng.uniform(0, 1, len(cell)) < density]
    pts = ((cell + rng.uniform(0.1, 0.9, cell.shape)) * 0.05).astype(np.float32)
    om = orc.OracleMap(dims, (0.0, 0.0, 0.0), 0.05)
    om.integrate(pts, POSE)
    ores = om.segment(orc.make_params(n_hyp=8, classify=0, **kw))
    monkeypatch.setenv("VOXMPS_PAIR_CAP", str(cap))
    gm = vm.VoxelMap(dims, (0.0, 0.0, 0.0), 0.05)
    monkeypatch.delenv("VOXMPS_PAIR_CAP")
    gm.integrate(pts, POSE)
    for _ in range(2):  # the second time with the scratch that the first one grew
        gres = gm.segment(vm.segment_params(n_hyp=8, classify=0, **kw))
        compare_labels(gm.export_labels(), ores["voxels"])
        compare_planes(gres, ores, gm.export_clusters(), check_refit=False)
