"""What a tree cannot be built from, and trees damaged after their build: the
status word reports them, and nothing outside the tree's arrays is touched."""
import numpy as np
import pytest

from gpu_util import device, og, torch

pytestmark = pytest.mark.gpu

ETREE = 5


def _particles(n, seed):
    dev = device()
    g = torch.Generator(dev).manual_seed(seed)
    return torch.rand((n, 3), dtype=torch.float64, device=dev, generator=g)


@pytest.mark.parametrize("n", [33, 513, 20000])
@pytest.mark.parametrize("how", ["descending", "one swap", "64 bits"])
def test_tree_refuses_keys_out_of_order(n, how):
    """Keys that are not ascending, or have a 64th bit (a root of sixteen
    octants), give OG_ETREE and NaN forces."""
    m = og()
    p = _particles(n, n)
    mass = torch.ones(n, dtype=torch.float64, device=p.device)
    keys, order = m.keys_sort(p, 1.0)
    if how == "descending":
        keys = keys.flip(0).contiguous()
    elif how == "one swap":
        keys[n // 2 - 1:n // 2 + 1] = keys[n // 2 - 1:n // 2 + 1].flip(0)
    else:
        keys = torch.tensor(np.sort(keys.cpu().numpy().view(np.uint64) << np.uint64(1)).view(np.int64), device=p.device)
    tree = m.tree_build(keys, order, p, mass, 1e-3, 1.0, check=False)
    assert m.poll_status(tree.mem) == ETREE
    out = torch.zeros((n, 3), device=p.device)
    with pytest.raises(m.OGError) as e:
        m.shortrange_accel(tree, 0.05, 0.5, out=out)
    assert e.value.code == ETREE and torch.isnan(out).all()


def _orders(tree, n):
    """The walks' two orders of the groups inside the tree buffer, which ends
    with them, their buckets and the topology passes' block counts."""
    up = lambda b: -(-b // 256) * 256  # noqa: E731
    g = -(-n // 32)
    end = og().lib().og_tree_bytes(n, None) - up(4 * 22 * -(-n // 512)) - 2 * up(g)
    at = [end - 2 * up(4 * g), end - up(4 * g)]
    out = [tree.mem[a:a + 4 * g].view(torch.int32) for a in at]
    for o in out:
        assert torch.equal(o.sort().values, torch.arange(g, dtype=torch.int32, device=o.device))
    return out


@pytest.mark.parametrize("n", [65, 5000, 32 * 24576])
@pytest.mark.parametrize("value", [-1, "groups", -(1 << 31), (1 << 31) - 1])
def test_damaged_order_is_reported(n, value):
    """An entry of the walks' order that is no group is reported, not followed."""
    m = og()
    p = _particles(n, 7)
    keys, order = m.keys_sort(p, 1.0)
    tree = m.tree_build(keys, order, p, torch.ones(n, dtype=torch.float64, device=p.device), 1e-3 * n ** (-1 / 3), 1.0)
    r_s = min(0.1, 0.3 * n ** (-1 / 3))
    w = torch.ones((n, 3), device=p.device)
    for o in _orders(tree, n):
        o[o.shape[0] // 2] = o.shape[0] if value == "groups" else value
    for call in (lambda: m.shortrange_accel(tree, r_s, 0.5), lambda: m.shortrange_accel(tree, r_s, 0.5, prec="fp64"),
                 lambda: m.shortrange_adjoint(tree, r_s, 0.5, w),
                 lambda: m.shortrange_accel_adjoint(tree, r_s, 0.5, w), lambda: m.sph_density(tree, 32)):
        with pytest.raises(m.OGError) as e:
            call()
        assert e.value.code == ETREE
    # walks over ranges go in tree order and do not read it
    g = int(tree.header.n_groups)
    out = torch.full((n, 3), float("nan"), device=p.device)
    m.shortrange_accel(tree, r_s, 0.5, out=out, groups=(0, g // 2))
    m.shortrange_accel(tree, r_s, 0.5, out=out, groups=(g // 2, g))
    assert torch.isfinite(out).all()
