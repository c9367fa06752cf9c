"""The number of kernels each call is said to launch."""
import pytest

from gpu_util import device, og, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [4096, 16384, 16385, 60_000])
def test_launches_per_call(n):
    from torch.profiler import ProfilerActivity, profile
    dev = device()
    m = og()
    p = torch.rand((n, 3), dtype=torch.float64, device=dev, generator=torch.Generator(dev).manual_seed(n))
    mass = torch.ones(n, dtype=torch.float64, device=dev)
    keys, order = m.keys_sort(p, 1.0)
    tree = m.tree_build(keys, order, p, mass, 1e-4, 1.0)
    plan = m.PMPlan(32)
    acc, vel = torch.zeros((n, 3), device=dev), torch.zeros_like(p)
    calls = {"keys_sort": lambda: m.keys_sort(p, 1.0, check=False),
             "tree_build": lambda: m.tree_build(keys, order, p, mass, 1e-4, 1.0, check=False),
             "accel": lambda: m.shortrange_accel(tree, 0.02, 0.5, check=False),
             "adjoint": lambda: m.shortrange_adjoint(tree, 0.02, 0.5, acc, check=False),
             "sph": lambda: m.sph_density(tree, 32, check=False),
             "pm": lambda: m.pm_accel(plan, p, mass, 1.0, 0.04, check=False),
             "kick": lambda: m.kick(vel, acc, None, 0.1), "drift": lambda: m.drift(p, vel, 0.0)}
    for _ in range(2):  # the profiler's first session may come up empty
        with profile(activities=[ProfilerActivity.CUDA]):
            for call in calls.values():
                call()
            torch.cuda.synchronize()
    for name, call in calls.items():
        torch.cuda.synchronize()
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            call()
            torch.cuda.synchronize()
        ours = [e.name for e in prof.events() if "og::k_" in e.name]
        if not ours:
            pytest.skip("no device events from the profiler here")
        assert len(ours) == m.launches_per_call(n)[name], (name, ours)
    plan.close()
