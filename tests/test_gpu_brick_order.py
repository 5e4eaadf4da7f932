"""GPU: brick ordering at the edges of its tiles of 256 table entries (one
entry, a full tile, one more, more tiles than one look-back covers, most of
them empty) and the per-warp sums of integration over groups of every size,
against the oracle: integer sums and voxel order are exact."""
import numpy as np
import pytest

from parity import compare_sums

pytestmark = pytest.mark.gpu

POSE = np.array([1, 0, 0, 0, 0, 1, 0, 0, 0, 0, 1, 0], np.float32)


def _grouped(rng, ext, groups):
    """Points in runs and interleaved: a group is a place that gets `size` points."""
    pts = np.concatenate([np.repeat(rng.uniform(0, 1, (1, 3)) * ext, k, 0) for k in groups])
    pts = pts + rng.uniform(-1e-3, 1e-3, pts.shape)
    return np.concatenate([pts, pts[rng.permutation(len(pts))], pts[::7]]).astype(np.float32)


@pytest.mark.parametrize("bricks", [(1, 1, 1), (16, 16, 1), (257, 1, 1), (40, 41, 43)])
def test_order_and_sums(orc, bricks):
    from paper_2510_01592_gb300 import vm
    rng = np.random.default_rng(sum(bricks))
    dims = tuple(8 * b for b in bricks)
    ext = np.array(dims) * 0.005
    gm, om = vm.VoxelMap(dims, (0.0, 0.0, 0.0), 0.005), orc.OracleMap(dims, (0.0, 0.0, 0.0), 0.005)
    sizes = list(range(1, 34)) * 3 + [64, 100, 1, 1, 1, 2, 2, 31, 32, 33] + [1] * 64
    for n_groups in (1, len(sizes)):
        p = _grouped(rng, ext, sizes[-n_groups:])
        p[::11] = np.nan
        gm.integrate(p, POSE)
        om.integrate(p, POSE)
        compare_sums(gm, om)
