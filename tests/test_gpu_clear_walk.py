"""GPU: the two-part ray walk of Eq. 2 clearing at its edges, against the
oracle: rays along the axes and diagonals (ties), rays that end exactly on
voxel borders, that leave the grid, that stay in one voxel; odd grid sizes;
sensors on the grid's faces and corners; a scrolled window."""
import numpy as np
import pytest

from parity import compare_sums

pytestmark = pytest.mark.gpu


def _pose(t):
    return np.array([1, 0, 0, t[0], 0, 1, 0, t[1], 0, 0, 1, t[2]], np.float32)


def _rays(rng, ext, t, n):
    """End points relative to a sensor at t: random, out of the grid, on borders, along axes and diagonals."""
    e = rng.uniform(-0.3, 1.3, (n, 3)) * ext
    k = n // 5
    e[:k] = np.round(e[:k] / 0.05) * 0.05
    e[k:2 * k] = t
    e[np.arange(k, 2 * k), rng.integers(0, 3, k)] += rng.uniform(-1.0, 1.0, k) * ext.max()
    e[2 * k:3 * k] = t + rng.uniform(-1, 1, (k, 1)) * ext.max() * rng.choice([-1.0, 1.0], (k, 3))
    e[3 * k:3 * k + 8] = t + rng.uniform(-0.01, 0.01, (8, 3))
    return (e - t).astype(np.float32)


@pytest.mark.parametrize("dims", [(61, 47, 33), (8, 8, 8), (130, 3, 17)])
@pytest.mark.parametrize("scrolled", [False, True])
def test_walk_edges(orc, dims, scrolled):
    from paper_2510_01592_gb300 import vm
    rng = np.random.default_rng(sum(dims) + scrolled)
    ext = np.array(dims) * 0.05
    shift = np.array([3, -2, 1]) if scrolled else np.zeros(3, int)
    lo = shift * 8 * 0.05
    gm, om = vm.VoxelMap(dims, (0.0, 0.0, 0.0), 0.05), orc.OracleMap(dims, (0.0, 0.0, 0.0), 0.05)
    if scrolled:
        gm.scroll(shift)
        om.scroll(shift)
    fill = (lo + rng.uniform(0, 1, (4000, 3)) * ext).astype(np.float32)
    for t in (0.5 * ext, 0 * ext, np.float32(0.999) * ext, np.array([0.0, 0.5, 0.25]) * ext):
        gm.integrate(fill, _pose((0, 0, 0)))
        om.integrate(fill, _pose((0, 0, 0)))
        p, pose = _rays(rng, ext, t, 600), _pose(lo + t)
        gm.integrate(p, pose, clear=True)
        om.clear_rays(p, pose)
        om.integrate(p, pose)
        compare_sums(gm, om)
    assert gm.stats()["voxels_cleared"] > 0
