"""GPU: a thread's direct fits (vm_fit_planes) share one scratch and one result
block; calls of different shapes on one thread give the plan's outputs, and come
to rest: no more launches or allocations a call than the shape takes alone."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _clusters(k, n, seed):
    """k patches of n points, with outliers; offsets int32 [k + 1]."""
    import torch
    rng = np.random.default_rng(seed)
    p = rng.uniform(-0.5, 0.5, (k, n, 3)) * np.array([1, 1, 0.004]) + rng.uniform(-4, 4, (k, 1, 3))
    off = np.arange(0, k * n + 1, n, dtype=np.int32)
    return torch.from_numpy(p.reshape(-1, 3).astype(np.float32)).cuda(), torch.from_numpy(off).cuda()


def _cost(vm, call):
    """Launches and allocations of a call."""
    a = vm.launch_count(), vm.allocation_count()
    call()
    return vm.launch_count() - a[0], vm.allocation_count() - a[1]


def _in_thread(work):
    """Runs work in a thread of its own (the scratch is a thread's)."""
    import threading
    out = []

    def body():
        try:
            out.append(work())
        except BaseException as e:  # handed to the caller
            out.append(e)

    t = threading.Thread(target=body)
    t.start()
    t.join()
    if isinstance(out[0], BaseException):
        raise out[0]
    return out[0]


def test_alternating_shapes_come_to_rest():
    from paper_2510_01592_gb300 import vm
    prm, few, many, wide = vm.segment_params(seed=3), *(_clusters(16, 16000, 1), _clusters(2000, 50, 2)), _clusters(3, 64, 4)
    wide_prm = vm.segment_params(n_hyp=1024, seed=3)
    batches = [(few, prm), (many, prm), (wide, wide_prm)]

    def work():
        for (xyz, off), p in batches:
            vm.fit_planes(xyz, off, p)
        return [[_cost(vm, lambda: vm.fit_planes(xyz, off, p)) for (xyz, off), p in batches] for _ in range(3)]

    alone = [_in_thread(lambda: (vm.fit_planes(*b, p), _cost(vm, lambda: vm.fit_planes(*b, p)))[1]) for b, p in batches]
    assert all(a[1] == 0 for a in alone)
    assert _in_thread(work) == [alone] * 3


def test_hulls_past_the_result_block_are_packed_again_only():
    """The first call of a thread, with more hull vertices than its result block starts with (48 a cluster and 4096):
    the fit runs once."""
    import torch
    from paper_2510_01592_gb300 import vm
    k, n = 200, 20000
    rng = np.random.default_rng(7)
    r, a = np.sqrt(rng.random((k, n))), rng.random((k, n)) * 2 * np.pi
    p = np.stack([r * np.cos(a), r * np.sin(a), rng.normal(0, 0.001, (k, n))], -1).reshape(-1, 3).astype(np.float32)
    xyz = torch.from_numpy(p).cuda()
    off = torch.arange(0, k * n + 1, n, dtype=torch.int32, device="cuda")
    prm = vm.segment_params(n_hyp=32, seed=1)

    def work():
        first = _cost(vm, lambda: res.append(vm.fit_planes(xyz, off, prm)))
        return first[0], _cost(vm, lambda: res.append(vm.fit_planes(xyz, off, prm)))

    res = []
    first, second = _in_thread(work)
    assert len(res[0]["hull_xy"]) > 48 * k + 4096
    assert second[1] == 0 and first <= second[0] + 2  # the pack and its header
    want = vm.FitPlan(k, k * n, prm).run(xyz, off)
    for key in ("planes", "hull_xy", "hull_xyz"):
        assert res[0][key].tobytes() == res[1][key].tobytes() == want[key].tobytes(), key


def test_many_small_clusters_with_over_a_million_hull_vertices():
    from paper_2510_01592_gb300 import vm
    k = 150_000
    xyz, off = _clusters(k, 24, 5)
    prm = vm.segment_params(n_hyp=8, seed=2)
    got = _in_thread(lambda: vm.fit_planes(xyz, off, prm))
    assert len(got["hull_xy"]) > 1 << 20
    want = vm.FitPlan(k, k * 24, prm).run(xyz, off)
    for key in ("planes", "hull_xy", "hull_xyz"):
        assert got[key].tobytes() == want[key].tobytes(), key


def _same(a, b):
    return all(a[key].tobytes() == b[key].tobytes() for key in ("planes", "hull_xy", "hull_xyz"))


def test_direct_fits_take_the_kernels_for_the_points_they_have():
    """A large batch (over four million points) takes more kernels than a small one; small ones after it come back to
    their own within eight calls, and where the two alternate the large ones keep theirs.  The outputs are the same."""
    from paper_2510_01592_gb300 import vm
    small, large, prm = _clusters(16, 5000, 1), _clusters(40, 120000, 2), vm.segment_params(n_hyp=32, seed=3)

    def call(b, res=None):
        c = _cost(vm, lambda: (res if res is not None else []).append(vm.fit_planes(*b, prm)))
        return c[0]

    def work():
        res = []
        call(small)
        few = call(small, res)
        call(large)
        many = call(large, res)
        assert many > few
        after = [call(small, res) for _ in range(10)]
        assert after[-1] == few and _same(res[0], res[2]) and _same(res[0], res[-1])
        call(large)  # from here on in turn
        for _ in range(4):
            call(small)
            assert call(large, res) == many
        assert _same(res[1], res[-1])

    _in_thread(work)


def test_a_plan_takes_the_kernels_for_the_points_it_has():
    """Likewise a plan that is sized for more: and once both kinds of batch have run, none is captured again."""
    from paper_2510_01592_gb300 import vm
    small, large, prm = _clusters(16, 5000, 1), _clusters(40, 120000, 2), vm.segment_params(n_hyp=32, seed=3)
    plan, own = vm.FitPlan(40, 4_800_000, prm), vm.FitPlan(16, 80000, prm)
    want = own.run(*small)
    few = _cost(vm, lambda: own.run(*small))[0]
    for _ in range(10):
        assert _same(plan.run(*small), want)
    assert _cost(vm, lambda: plan.run(*small))[0] == few
    first = plan.run(*large)
    many = _cost(vm, lambda: plan.run(*large))[0]
    assert many > few
    captures = vm.capture_count()
    for _ in range(10):
        assert _same(plan.run(*large), first)
        assert _cost(vm, lambda: plan.run(*large))[0] == many
    assert vm.capture_count() == captures
