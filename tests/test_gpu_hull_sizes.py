"""GPU: the hull kernel at the numbers of survivors where its passes change (all
points of a ring survive the first filter), against the oracle bit for bit:
none to few, one pass of few or many directions, a second pass, more than the
shared-memory sort holds; with points inside, repeated points, a long arc over
a far point, and a line."""
import numpy as np
import pytest

from parity import compare_planes

pytestmark = pytest.mark.gpu


def _ring(rng, n, kind):
    a = np.sort(rng.uniform(0, 2 * np.pi, n))
    if kind == "arc":  # an arc over a far point
        a = np.pi * np.arange(n) / max(n - 1, 1)
    r = 0.7 * (1 + (0.03 * rng.uniform(-1, 1, n) if kind == "rough" else 0))
    p = np.stack([r * np.cos(a), r * np.sin(a), np.zeros(n)], 1)
    if kind == "arc":
        p = np.concatenate([p, [[0.9, -3.0, 0.0]]])
    if kind == "line":
        p[:, 1] = p[:, 0]
    inner = p[:, None, :] * rng.uniform(0, 0.9, (len(p), 3, 1))
    return np.concatenate([p, inner.reshape(-1, 3), p[::5]]) + [1.0, -2.0, 0.5]


@pytest.mark.parametrize("kind", ["smooth", "rough", "arc", "line"])
def test_hull_sizes(orc, kind):
    import torch
    from paper_2510_01592_gb300 import vm
    rng = np.random.default_rng(len(kind))
    sizes = (3, 5, 31, 64, 79, 80, 81, 95, 96, 97, 128, 129, 133, 134, 160, 161, 255, 256, 257, 426, 427, 512, 513, 700,
             1706, 1707, 2049, 2600)
    cl = [_ring(rng, n, kind).astype(np.float32) for n in sizes]
    off = np.r_[0, np.cumsum([len(c) for c in cl])].astype(np.uint32)
    xyz = np.concatenate(cl)
    ores = orc.fit_planes(xyz, off, orc.make_params(n_hyp=16, seed=2))
    gres = vm.fit_planes(torch.from_numpy(xyz).cuda(), torch.from_numpy(off.astype(np.int32)).cuda(),
                         vm.segment_params(n_hyp=16, seed=2))
    compare_planes(gres, ores, check_refit=False)
