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
