"""GPU: the large-fit scoring (bounded tiles, dropped hypotheses) against the
small-fit scoring, which makes every test: a plan sized for five million points
takes the former, one sized for the batch the latter; every output is equal bit
for bit.  Clusters at the edges of a tile and of a chunk, empty and tiny ones,
repeated and collinear points, points that are not numbers, clusters far from
the origin, thin and thick ones; one to 1024 hypotheses; thresholds from zero
to one that takes everything."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _clusters(rng):
    out = []
    for n in (0, 1, 2, 3, 4, 63, 64, 65, 255, 256, 257, 2047, 2048, 2049, 4097, 30001):
        side = max(1, int(np.sqrt(n)))
        i = np.arange(n)
        p = np.stack([i % side * 0.01, i // side * 0.01, rng.normal(0, 0.001, n)], 1)
        q, _ = np.linalg.qr(rng.normal(size=(3, 3)))
        p = p @ q + rng.uniform(-8, 8, 3)
        k = n // 20
        if k:
            at = rng.choice(n, k, replace=False)
            p[at] = rng.uniform(p.min(0) - 0.05, p.max(0) + 0.05, (k, 3))
        out.append(p)
    out.append(np.tile(rng.uniform(-1, 1, 3), (500, 1)))                                  # one point, repeated
    out.append(np.linspace(0, 1, 700)[:, None] * rng.uniform(-1, 1, 3))                   # a line
    out.append(rng.uniform(-1, 1, (5000, 3)))                                             # no plane
    out.append(out[13] + 100.0)                                                           # far away: coarse coordinates
    out.append(out[14] * np.array([1.0, 1.0, 8.0]))                                       # thick
    bad = out[14].copy()
    bad[::97] = np.nan
    bad[50::311, 1] = np.inf
    out.append(bad)
    order = rng.permutation(out[15].shape[0])
    out.append(out[15][order])                                                            # points in no order
    return out


@pytest.mark.parametrize("hyps,eps", [(100, 0.01), (1, 0.01), (7, 0.0), (256, 0.002), (1024, 0.03), (64, 50.0)])
def test_large_fit_scoring_equals_the_small_one(hyps, eps):
    import torch
    from paper_2510_01592_gb300 import vm
    cl = _clusters(np.random.default_rng(hyps))
    off = np.r_[0, np.cumsum([len(c) for c in cl])].astype(np.int32)
    xyz = torch.from_numpy(np.concatenate(cl).astype(np.float32)).cuda()
    d_off = torch.from_numpy(off).cuda()
    prm = vm.segment_params(n_hyp=hyps, eps=eps, seed=5)
    small = vm.FitPlan(len(cl), int(off[-1]), prm).run(xyz, d_off)
    large = vm.FitPlan(len(cl), 5_000_000, prm)
    for tuning in (None, (256, 4, 4), (4096, 8, 2), (1024, 1, 3)):
        if tuning and -(-hyps // tuning[1]) <= 256:
            large.set_tuning(*tuning)
        got = large.run(xyz, d_off)
        for key in ("planes", "hull_xy", "hull_xyz"):
            a, b = small[key], got[key]
            assert a.shape == b.shape and a.tobytes() == b.tobytes(), (key, tuning)
