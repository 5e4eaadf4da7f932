"""GPU: the large-fit scoring where a reference plane's normal is no unit vector:
its samples lie so close together that the squared length of their cross
product is a subnormal number of a few bits.  The cluster is a flat patch with a
dense spot at the origin and a few points just off the patch; the oracle's
selected hypothesis and count, and every output of the small-fit scoring, which
makes every test."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _patch(seed):
    rng = np.random.default_rng(seed)
    spot, wide = np.zeros((150, 3)), np.zeros((100, 3))
    spot[:, :2] = rng.uniform(-1, 1, (150, 2)) * 7e-12
    wide[:, 0], wide[:, 1] = rng.uniform(-0.5, 0.5, 100), rng.uniform(-0.2, 0.2, 100)
    wide[:8, 0], wide[:8, 1] = 0.5, rng.uniform(-0.02, 0.02, 8)
    wide[8:16, 0] = -0.5
    wide[16], wide[17] = (0.0, 0.7, 0.0), (0.0, -0.69, 0.0)
    off = np.tile([0.5, 0.0, 0.014], (6, 1))
    off[:, 1] = rng.uniform(-0.01, 0.01, 6)
    return np.concatenate([spot, wide, off]).astype(np.float32)[rng.permutation(256)]


@pytest.mark.parametrize("seed", [0, 10, 26, 31, 42])
def test_scoring_with_a_reference_normal_that_is_no_unit_vector(orc, seed):
    import torch
    from paper_2510_01592_gb300 import vm
    p = _patch(seed)
    counts, _, best = orc.ransac_counts(p, 0, 256, seed, 0.01)
    xyz, off = torch.from_numpy(p).cuda(), torch.tensor([0, len(p)], dtype=torch.int32, device="cuda")
    prm = vm.segment_params(n_hyp=256, seed=seed)
    small = vm.FitPlan(1, len(p), prm).run(xyz, off)
    large = vm.FitPlan(1, 5_000_000, prm).run(xyz, off)
    for got in (small, large):
        assert (got["planes"]["best_h"][0], got["planes"]["inlier_count"][0]) == (best, counts[best])
    for key in ("planes", "hull_xy", "hull_xyz"):
        assert small[key].tobytes() == large[key].tobytes(), key
