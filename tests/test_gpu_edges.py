"""Sizes at which the sort, the tree build and the walks change path: tile and
block edges of the sort and the topology passes, one to four warps a group, a
ragged last group, coincident particles down to the last level."""
import numpy as np
import pytest

import ics
from gpu_util import GRAD_TOL, device, grad_scaled_err, og, torch

pytestmark = pytest.mark.gpu


def _case(n, seed, clumps=0):
    rng = np.random.default_rng(seed)
    pos = rng.random((n, 3))
    if clumps:  # exact duplicates, more than a leaf of each: leaves of the last level
        pos[: n // 2] = pos[rng.integers(0, clumps, n // 2)]
    return pos, 0.5 + rng.random(n), np.full(n, 0.3 * n ** (-1 / 3))


@pytest.mark.parametrize("n", [1, 511, 512, 513, 4095, 4096, 4097, 8193, 1024 * 32, 1024 * 32 + 1, 4096 * 32 + 33])
@pytest.mark.parametrize("clumps", [0, 5])
def test_sort_tree_and_walks(orc, n, clumps):
    dev = device()
    m = og()
    pos, mass, eps = _case(n, n + clumps, clumps if n > 400 else 0)
    p, mt, e = (torch.tensor(x, dtype=torch.float64, device=dev) for x in (pos, mass, eps))
    keys, order = m.keys_sort(p, 1.0)
    ks, o = orc.sort(orc.keys(pos, 1.0)[0])
    assert np.array_equal(keys.cpu().numpy().view(np.uint64), ks) and np.array_equal(order.cpu().numpy(), o)
    tree = m.tree_build(keys, order, p, mt, e, 1.0)
    r_s = min(0.1, 0.7 * n ** (-1 / 3))
    T = orc.Tree(pos, mass, 2.8 * eps, leaf_size=16)
    assert tree.node_count() == T.nodes()["level"].shape[0]
    tg = np.unique(np.concatenate([np.arange(max(0, n - 40), n), np.linspace(0, n - 1, 300).astype(int)]))
    ref, cnt = T.walk(r_s, 4.5 * r_s, 0.5, targets=tg)
    scale = max(np.sqrt((ref ** 2).sum(1).mean()), 1e-300)
    # FP32 terms are good to about 2e-6 and FP64 ones to a few ulp; a target's
    # error is that of its largest terms (close pairs), within 10 rms here
    for prec, tol in (("fp32", 2e-5), ("fp64", 1e-13)):
        acc, total, c = m.shortrange_accel(tree, r_s, 0.5, prec=prec, counts=True)
        assert np.array_equal(c.cpu().numpy()[tg], cnt)
        assert int(total.item()) == int(c.sum().item())
        assert np.abs(acc.double().cpu().numpy()[tg] - ref).max() <= tol * max(scale, np.abs(ref).max())
    # a range of groups gives the full walk's sums, and the fused walk the forward's
    acc, total, _ = m.shortrange_accel(tree, r_s, 0.5)
    part = torch.zeros_like(acc)
    g = int(tree.header.n_groups)
    for a, b in ((0, g // 3), (g // 3, g)):
        m.shortrange_accel(tree, r_s, 0.5, out=part, groups=(a, b))
    assert torch.equal(acc, part)
    w = torch.tensor(ics.loss_weights(n, 5), dtype=torch.float32, device=dev)
    fa, ft, _, dx, dm = m.shortrange_accel_adjoint(tree, r_s, 0.5, w)
    assert torch.equal(fa, acc) and int(ft.item()) == int(total.item())
    if n <= 8193:
        s = tg[:: max(1, len(tg) // 60)]
        gp, gm, sp, sm = T.adjoint(r_s, 4.5 * r_s, 0.5, w.double().cpu().numpy(), s, with_scale=True)
        assert grad_scaled_err(dx.cpu().numpy()[s], gp, sp) < GRAD_TOL
        assert grad_scaled_err(dm.cpu().numpy()[s], gm, sm) < GRAD_TOL


@pytest.mark.parametrize("n", [16385, 17 * 1024 - 1, (1 << 18) - 1, 1 << 18, (1 << 18) + 1])
def test_sort_tile_sizes(orc, n):
    """Either side of the key counts at which the tiles of the sort change size."""
    pos = np.random.default_rng(n).random((n, 3))
    pos[: n // 4] = pos[0]  # one digit that fills whole tiles
    keys, order = og().keys_sort(torch.tensor(pos, dtype=torch.float64, device=device()), 1.0)
    ks, o = orc.sort(orc.keys(pos, 1.0)[0])
    assert np.array_equal(keys.cpu().numpy().view(np.uint64), ks) and np.array_equal(order.cpu().numpy(), o)


@pytest.mark.parametrize("room,n", [((1 << 18) + 1, 1 << 18), (290_000, 235_000), ((1 << 18) + 1, 16384)])
def test_sort_in_a_larger_workspace(orc, room, n):
    """A workspace sized for more keys, in tiles of the other size, serves fewer."""
    dev = device()
    m = og()
    ws = m._workspace(m.lib().og_keys_sort_ws_bytes(room), dev)
    pos = np.random.default_rng(n).random((n, 3))
    keys, order = m.keys_sort(torch.tensor(pos, dtype=torch.float64, device=dev), 1.0, ws=ws)
    ks, o = orc.sort(orc.keys(pos, 1.0)[0])
    assert np.array_equal(keys.cpu().numpy().view(np.uint64), ks) and np.array_equal(order.cpu().numpy(), o)


@pytest.mark.parametrize("axis", ["random", "ones"])
def test_keys_by_table_and_by_bits(axis):
    """Keys of more than 16,384 particles are looked up level by level, fewer
    are computed bit by bit: the same numbers, over all bits of the cell."""
    dev = device()
    m = og()
    rng = np.random.default_rng(3)
    cell = rng.integers(0, 1 << 21, (3 * 16384, 3))
    if axis == "ones":  # long runs of equal bits, from either end
        cell = (1 << 21) - (1 << rng.integers(0, 22, (3 * 16384, 3)))
        cell[::2] ^= (1 << 21) - 1
        cell = np.clip(cell, 0, (1 << 21) - 1)
    pos = torch.tensor((cell + 0.5) * 2.0 ** -21, dtype=torch.float64, device=dev)
    keys, _ = m.keys_sort(pos, 1.0)
    parts = torch.cat([m.keys_sort(p.contiguous(), 1.0)[0] for p in pos.split(16384)])
    assert torch.equal(keys, parts.sort().values)


def _nodes_of(keys, leaf):
    """The nodes over sorted keys, level by level in key order, by their definition."""
    n = keys.shape[0]
    first, count, parent = np.array([0]), np.array([n]), np.array([-1])
    out, base = [], 0
    for level in range(22):
        split = (count > leaf) & (level < 21)
        out.append([np.full_like(first, level), first, count, parent, split])
        if not split.any():
            break
        pre = keys >> np.uint64(63 - 3 * (level + 1))
        starts = np.flatnonzero(np.concatenate([[True], pre[1:] != pre[:-1]]))
        ends = np.concatenate([starts[1:], [n]])
        own = np.searchsorted(first, starts, "right") - 1  # the node of this level that a run may lie in
        keep = (own >= 0) & split[own] & (starts < first[own] + count[own])
        parent = base + own[keep]
        base += first.shape[0]
        first, count = starts[keep], (ends - starts)[keep]
    level, first, count, parent, split = (np.concatenate([o[i] for o in out]) for i in range(5))
    nchild = np.bincount(parent[1:], minlength=level.shape[0])
    child = np.full(level.shape[0], -1)
    child[parent[1:][::-1]] = np.arange(1, level.shape[0])[::-1]
    return dict(level=level, first=first, count=count, parent=parent, nchild=nchild, child_first=child)


@pytest.mark.parametrize("n,leaf,clumps", [(511, 16, 0), (5000, 1, 7), (40_000, 1, 0), (40_000, 32, 5), (70_001, 15, 3),
                                           (70_001, 16, 3), (512 * 1024 + 17, 16, 0), (4_300_000, 16, 2)])
def test_nodes_of_many_blocks(n, leaf, clumps):
    """Node ranges and links over the blocks of the topology passes, runs that
    span many of them, up to more blocks than one step of their scan takes."""
    dev = device()
    m = og()
    pos, mass, eps = _case(n, n + leaf, clumps)
    p, mt, e = (torch.tensor(x, dtype=torch.float64, device=dev) for x in (pos, mass, eps))
    keys, order = m.keys_sort(p, 1.0)
    got = m.tree_build(keys, order, p, mt, e, 1.0, p=m.params(leaf_size=leaf, node_capacity=4 * n + 1024)).nodes()
    for k, v in _nodes_of(keys.cpu().numpy().view(np.uint64), leaf).items():
        assert np.array_equal(got[k].cpu().numpy(), v), k


@pytest.mark.parametrize("n", [31, 1024 * 32 - 1, 3 * 1024 * 32 + 1])
def test_orders_hold_every_group(n):
    """The walks' orders of the groups (tiles of 1024 groups, buckets of
    estimated work): a full walk leaves no target out in either precision and
    agrees with walks over ranges, which go in tree order; SPH likewise."""
    dev = device()
    m = og()
    rng = np.random.default_rng(n)
    pos = rng.random((n, 3))
    pos[: n // 2] = np.mod(0.98 + 0.01 * rng.standard_normal((n // 2, 3)), 1.0)  # a clump across the box's corner
    p = torch.tensor(pos, dtype=torch.float64, device=dev)
    keys, order = m.keys_sort(p, 1.0)
    tree = m.tree_build(keys, order, p, torch.ones(n, dtype=torch.float64, device=dev), 0.3 * n ** (-1 / 3), 1.0)
    r_s = min(0.1, 0.625 * n ** (-1 / 3))
    g = int(tree.header.n_groups)
    for prec in ("fp32", "fp64"):
        full = torch.full((n, 3), float("nan"), dtype=torch.float32 if prec == "fp32" else torch.float64, device=dev)
        part = full.clone()
        m.shortrange_accel(tree, r_s, 0.5, prec=prec, out=full)
        for a, b in ((0, g // 2), (g // 2, g)):
            if b > a:
                m.shortrange_accel(tree, r_s, 0.5, prec=prec, out=part, groups=(a, b))
        assert torch.isfinite(full).all() and torch.equal(full, part)
    if n > 100:
        h, rho, ngb = m.sph_density(tree, 32)
        assert (h > 0).all() and (rho > 0).all() and (ngb > 0).all()


@pytest.mark.parametrize("n,n_ngb", [(97, 16), (129, 16), (1024 * 32, 32), (1024 * 32 + 5, 100)])
def test_sph_sizes(n, n_ngb):
    """SPH at few particles, one against four warps a group, more neighbours
    than a list holds, in a set with denser clumps; h and rho as in
    test_gpu_sph.py (float-float distances, second-order steps up to 3e-4)."""
    from oracle import og_sph as S
    dev = device()
    m = og()
    rng = np.random.default_rng(n)
    pos = rng.random((n, 3))
    pos[: n // 2] = np.mod(0.5 + 0.02 * rng.standard_normal((n // 2, 3)), 1.0)
    mass = 0.5 + rng.random(n)
    p, mt = (torch.tensor(x, dtype=torch.float64, device=dev) for x in (pos, mass))
    keys, order = m.keys_sort(p, 1.0)
    h, rho, ngb = m.sph_density(m.tree_build(keys, order, p, mt, 1e-3, 1.0), n_ngb)
    tg = np.linspace(0, n - 1, min(n, 60)).astype(int)
    ho = S.smoothing_length(pos, 1.0, n_ngb, targets=tg)
    np.testing.assert_allclose(h.cpu().numpy()[tg], ho, rtol=1e-9)
    np.testing.assert_allclose(rho.cpu().numpy()[tg], S.density(pos, mass, ho, 1.0, targets=tg), rtol=1e-9)
    cnt = [int((S.distances(pos, int(i), 1.0) < ho[k]).sum()) - 1 for k, i in enumerate(tg)]
    np.testing.assert_array_equal(ngb.cpu().numpy()[tg], cnt)


@pytest.mark.parametrize("groups", [24575, 24576, 24577])
def test_walk_of_many_groups(groups):
    """Either side of the group count from which the forward walk runs in
    blocks of one warp, the last group ragged: the sums of the walk in both
    directions at once, which goes in blocks of two at any size."""
    dev = device()
    m = og()
    n = 32 * groups - 31
    p = torch.rand((n, 3), dtype=torch.float64, device=dev, generator=torch.Generator(dev).manual_seed(groups))
    p[: n // 8] = (0.5 + 0.05 * (p[: n // 8] - 0.5)).contiguous()
    keys, order = m.keys_sort(p, 1.0)
    tree = m.tree_build(keys, order, p, torch.ones(n, dtype=torch.float64, device=dev), 0.05 * n ** (-1 / 3), 1.0)
    r_s = 0.625 * n ** (-1 / 3)
    acc, total, counts = m.shortrange_accel(tree, r_s, 0.5, counts=True)
    both, total2, counts2, _, _ = m.shortrange_accel_adjoint(tree, r_s, 0.5, torch.ones_like(acc), counts=True)
    assert torch.isfinite(acc).all() and torch.equal(acc, both)
    assert torch.equal(counts, counts2) and int(total.item()) == int(total2.item()) == int(counts.sum().item())


@pytest.mark.parametrize("n,N", [(300, 16), (20000, 32)])
def test_stepper_mesh_beside_tree(n, N):
    """Forces with the mesh on its own stream, from the default stream and from
    another one, against the calls one after the other.  The mesh sums its
    deposits in any order: a few FP32 rounding errors of the largest force."""
    dev = device()
    m = og()
    rng = np.random.default_rng(n)
    p = torch.tensor(rng.random((n, 3)), dtype=torch.float64, device=dev)
    S = m.TreePMStepper(p, torch.zeros_like(p), torch.full((n,), 1.0 / n, dtype=torch.float64, device=dev), 1e-3, 1.0,
                        0.7 * n ** (-1 / 3), 0.5, N)
    short, long = S.acc_s.clone(), S.acc_l.clone()  # the constructor's, checked one by one
    other = torch.cuda.Stream()
    other.wait_stream(torch.cuda.current_stream())
    for stream in (None, other):
        for _ in range(3):
            S.acc_s.fill_(float("nan"))
            S.acc_l.fill_(float("nan"))
            torch.cuda.synchronize()
            S.forces(stream=stream)
            S.poll(stream)
            assert torch.equal(S.acc_s, short)
            assert (S.acc_l - long).abs().max() <= 1e-5 * long.abs().max()
    p[n // 2, 1] = float("nan")
    with pytest.raises(m.OGError):
        S.step(0.0)
    S.close()


def _mesh_ref(pos, mass, N, r_s):
    """The mesh force in torch FP64 on the device (unit box)."""
    dev = pos.device
    u = pos * N
    i0 = torch.floor(u).long()
    f = u - i0
    w = [(1 - f[:, a], f[:, a]) for a in range(3)]
    rho = torch.zeros(N ** 3, dtype=torch.float64, device=dev)
    nodes = []
    for o in range(8):
        b = (o >> 2, (o >> 1) & 1, o & 1)
        i = [(i0[:, a] + b[a]) % N for a in range(3)]
        nodes.append(((i[0] * N + i[1]) * N + i[2], w[0][b[0]] * w[1][b[1]] * w[2][b[2]]))
        rho.index_add_(0, nodes[-1][0], mass * nodes[-1][1])
    hat = torch.fft.rfftn(rho.view(N, N, N))
    del rho
    k = torch.fft.fftfreq(N, 1.0 / N, dtype=torch.float64, device=dev)
    kz = torch.arange(N // 2 + 1, dtype=torch.float64, device=dev)
    for x in range(N):  # plane by plane: the largest mesh has 10^9 nodes
        k2 = (2 * np.pi) ** 2 * (k[x] ** 2 + k[:, None] ** 2 + kz[None, :] ** 2)
        S = (torch.sinc(k[x] / N) * torch.sinc(k / N)[:, None] * torch.sinc(kz / N)[None, :]) ** 4
        g = -4 * np.pi * torch.exp(-k2 * r_s ** 2) / (k2 * S) * N ** 3
        if x == 0:
            g[0, 0] = 0.0
        hat[x] *= g
    phi = torch.fft.irfftn(hat, s=(N, N, N))
    del hat
    acc = torch.zeros_like(pos)
    st = (N * N, N, 1)
    for j, wt in nodes:
        c = [j // (N * N), (j // N) % N, j % N]
        for a in range(3):
            v = [phi.view(-1)[j + ((c[a] + s) % N - c[a]) * st[a]] for s in (-2, -1, 1, 2)]
            acc[:, a] -= wt * N * ((2 / 3) * (v[2] - v[1]) - (1 / 12) * (v[3] - v[0]))
    return acc


@pytest.mark.parametrize("N", [8, 12, 16, 32, 64, 100, 128, 256, 512, 1024])
def test_pm_mesh_sides(N):
    """Every side's transform path (3-D, or planes and the fused x pass), with
    particles beside every face; bounds of test_gpu_pm.py."""
    dev = device()
    m = og()
    rng = np.random.default_rng(N)
    pos = rng.random((3000, 3))
    pos[:600] = np.mod(rng.normal(scale=1.5 / N, size=(600, 3)), 1.0)
    pos[600:900, 2] = np.mod(rng.normal(scale=2.0 / N, size=300), 1.0)
    p = torch.tensor(pos, dtype=torch.float64, device=dev)
    mt = torch.tensor(0.5 + rng.random(3000), dtype=torch.float64, device=dev)
    plan = m.PMPlan(N)
    a = m.pm_accel(plan, p, mt, 1.0, 1.25 / N).double()
    ref = _mesh_ref(p, mt, N, 1.25 / N)
    d = (a - ref).norm(dim=1)
    scale = ref.square().sum(1).mean().sqrt()
    plan.close()
    assert float(d.square().mean().sqrt() / scale) < 5e-6 and float(d.max() / scale) < 5e-5


def _fp64_case(rcut, side, seed, n=400):
    """Particles in a box of the given side whose mean spacing is far below the
    cut of rcut times r_s, which stays below half the box."""
    rng = np.random.default_rng(seed)
    return rng.random((n, 3)) * side, 0.5 + rng.random(n), np.full(n, 0.01 * side), 0.45 * side / rcut


@pytest.mark.parametrize("rcut,side", [(6.0, 1.0), (8.0, 1.0), (8.0, 50.0), (4.5, 2.0 ** 60), (4.5, 2.0 ** -60)])
def test_fp64_walk_beyond_its_table(orc, rcut, side):
    """The FP64 pair force where the short-range factor's table ends (u = 2.25, a
    cut of 4.5 r_s) and CUDA's functions take over, and in boxes whose squared
    distances leave the range of the reciprocal root's FP32 start.  Bound of
    test_sort_tree_and_walks."""
    dev = device()
    m = og()
    pos, mass, eps, r_s = _fp64_case(rcut, side, int(rcut * 10))
    p, mt, e = (torch.tensor(x, dtype=torch.float64, device=dev) for x in (pos, mass, eps))
    keys, order = m.keys_sort(p, side)
    tree = m.tree_build(keys, order, p, mt, e, side, p=m.params(rcut_factor=rcut))
    acc, _, c = m.shortrange_accel(tree, r_s, 0.5, prec="fp64", counts=True)
    ref, cnt = orc.Tree(pos, mass, 2.8 * eps, box=side).walk(r_s, rcut * r_s, 0.5)
    assert np.array_equal(c.cpu().numpy(), cnt)
    if rcut > 4.5:  # pairs on both sides of the table's end
        d = np.abs(pos[:, None] - pos[None])
        d = np.minimum(d, side - d)
        u = np.sqrt((d ** 2).sum(2)) / (2 * r_s)
        assert (np.abs(u - 2.25) < 0.05).sum() > 20 and ((u > 2.3) & (u < rcut / 2)).sum() > 100
    assert np.abs(acc.cpu().numpy() - ref).max() <= 1e-13 * np.abs(ref).max()


@pytest.mark.parametrize("n,N", [(500, 16), (30_000, 48)])
def test_stepper_in_a_graph(n, N):
    """A captured step (the mesh's fork and join become branches of the graph)
    replayed gives the states of uncaptured steps, whose mesh sums its deposits
    in any order: a few FP32 rounding errors of the largest force."""
    dev = device()
    m = og()
    rng = np.random.default_rng(n)
    x0 = torch.tensor(rng.random((n, 3)), dtype=torch.float64, device=dev)
    mass = torch.full((n,), 1.0 / n, dtype=torch.float64, device=dev)
    dt, steps = 1e-3, 3
    S, G = (m.TreePMStepper(x0.clone(), torch.zeros_like(x0), mass, 1e-3, 1.0, 0.7 * n ** (-1 / 3), 0.5, N)
            for _ in range(2))
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        G.step(dt, check=False)
    for _ in range(steps):
        S.step(dt)
        graph.replay()
    torch.cuda.synchronize()
    G.poll()
    amax = max(float(S.acc_s.abs().max()), float(S.acc_l.abs().max()))
    assert (G.vel - S.vel).abs().max() <= 1e-5 * amax * dt * steps
    assert (G.pos - S.pos).abs().max() <= 1e-5 * amax * dt * dt * steps * steps + 1e-15
    S.close()
    G.close()
