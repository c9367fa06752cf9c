"""A weight that is not finite, and a mass that overflows FP32, reach the
particles within the cut of theirs and no others."""
import numpy as np
import pytest

from gpu_util import device, og, torch

pytestmark = pytest.mark.gpu

R_S = 0.03  # a cut of 0.135


def _set(n, seed):
    dev = device()
    rng = np.random.default_rng(seed)
    pos = rng.random((n, 3))
    pos[: n // 4] = np.mod(0.02 * rng.standard_normal((n // 4, 3)), 1.0)  # a clump across the box's corner
    bad = n // 8
    d = pos - pos[bad]
    d -= np.rint(d)
    far = torch.tensor((d ** 2).sum(1) > (4.5 * R_S * 1.0001) ** 2, device=dev)
    t = lambda x: torch.tensor(x, dtype=torch.float64, device=dev)  # noqa: E731
    return t(pos), t(0.5 + rng.random(n)), bad, far


def _tree(pos, mass):
    m = og()
    keys, order = m.keys_sort(pos, 1.0)
    return m.tree_build(keys, order, pos, mass, 1e-3, 1.0)


def _same(a, b, far):
    a, b = a.double()[far], b.double()[far]
    assert torch.isfinite(a).all()
    assert (a - b).abs().max() <= 1e-5 * b.abs().max()  # other roundings of the same FP32 terms (2e-6 each)


@pytest.mark.parametrize("n", [3000, 200_000])
@pytest.mark.parametrize("value", [float("nan"), float("inf"), -float("inf"), 3e38])
def test_weight_stays_within_the_cut(n, value):
    m = og()
    pos, mass, bad, far = _set(n, n)
    assert 100 < int(far.sum()) < n - 100
    tree = _tree(pos, mass)
    w = torch.randn((n, 3), device=pos.device, generator=torch.Generator(pos.device).manual_seed(2))
    w[bad] = 0.0
    ref = m.shortrange_adjoint(tree, R_S, 0.5, w)
    w[bad, 1] = value
    for got in (m.shortrange_adjoint(tree, R_S, 0.5, w), m.shortrange_accel_adjoint(tree, R_S, 0.5, w)[3:5]):
        for a, b in zip(got, ref):
            _same(a, b, far)
    acc = m.shortrange_accel(tree, R_S, 0.5)[0]
    fused = m.shortrange_accel_adjoint(tree, R_S, 0.5, w)[0]
    assert (acc - fused).abs().max() <= 1e-5 * acc.abs().max()  # forces do not depend on the weights


@pytest.mark.parametrize("n", [3000, 200_000, 800_000])
def test_mass_stays_within_the_cut(n):
    m = og()
    pos, mass, bad, far = _set(n, n)
    ref = m.shortrange_accel(_tree(pos, mass), R_S, 0.5)[0]
    w = torch.ones((n, 3), device=pos.device)
    gref = m.shortrange_adjoint(_tree(pos, mass), R_S, 0.5, w)
    mass[bad] = 1e39
    tree = _tree(pos, mass)
    far_or_own = far.clone()
    far_or_own[bad] = True  # a particle's force does not hold its own mass
    _same(m.shortrange_accel(tree, R_S, 0.5)[0], ref, far_or_own)
    got = m.shortrange_accel_adjoint(tree, R_S, 0.5, w)
    _same(got[0], ref, far_or_own)
    for a, b in zip(got[3:5], gref):
        _same(a, b, far)
