"""What the library is timed on: whole passes through its public entry points.

A pass starts from the particles in their own order, as a simulation or a
fit has them at each step: keys and sort, tree, then the walk, its gradient,
the SPH density or the mesh.  The sets are those of the benchmark and the
tests (a uniform set, a Zel'dovich lattice, NFW haloes on a background, a
multi-mass zoom), drawn on the GPU from the seed.

exact() restates the method in plain torch FP64 (octree by Morton prefixes,
a breadth-first walk over (target, node) pairs, bisection for the SPH radius,
an FP64 mesh) and uses nothing of the library.
"""
from __future__ import annotations

import math

import torch

import paper_2606_17145_gb300 as og

LEAF = 16          # the library's default leaf size
RCUT = 4.5         # and its default cut, in units of r_s


def listed():
    return [
        # forces of a small set, as in a unit test, a few-body problem or one rank's share: launches and latency
        dict(name="forces_uniform_4096", kind="forces", set="uniform", n=4096, box=1.0, rs_cells=1.25, theta=0.5),
        # an early, near-homogeneous cosmological box
        dict(name="forces_lattice_128", kind="forces", set="lattice", n=128 ** 3, box=1.0, rs_cells=0.625, theta=0.5),
        # the benchmark's evolved box: 256^3 particles, most of them in haloes
        dict(name="forces_clustered_256", kind="forces", set="clustered", n=256 ** 3, box=1.0, rs_cells=0.625,
             theta=0.5),
        # a multi-mass zoom region in a box whose side is no power of two, a ragged count
        dict(name="forces_zoom_ragged", kind="forces", set="zoom", n=187_501, box=50.0, rs_cells=0.625, theta=0.5),
        # forward and backward through autograd on the clustered set: fitting a displacement field and masses
        dict(name="grad_clustered_128", kind="grad", set="clustered", n=128 ** 3, box=1.0, rs_cells=0.625, theta=0.5),
        # the same fit with loss weights known beforehand, on a lattice with an odd side
        dict(name="linear_loss_lattice_97", kind="linear_loss", set="lattice", n=97 ** 3, box=1.0, rs_cells=0.625,
             theta=0.5),
        # the all-FP64 walk: checking a run, or a problem that needs FP64 forces
        dict(name="fp64_clustered_64", kind="forces64", set="clustered", n=64 ** 3, box=1.0, rs_cells=0.625,
             theta=0.5),
        # keys and sort alone: a reordering or a domain decomposition, an odd count
        dict(name="keys_clustered_5m", kind="keys", set="clustered", n=5_000_011, box=1.0),
        # the long-range mesh at two cells a particle spacing
        dict(name="pm_lattice_128", kind="pm", set="lattice", n=128 ** 3, box=1.0, ngrid=256),
        # SPH densities of an evolved box
        dict(name="sph_clustered_128", kind="sph", set="clustered", n=128 ** 3, box=1.0, n_ngb=32),
        # SPH densities of a smaller smooth set, more neighbours, ragged, a box that is no power of two
        dict(name="sph_uniform_ragged", kind="sph", set="uniform", n=100_003, box=3.0, n_ngb=64),
        # one step of a TreePM simulation
        dict(name="kdk_lattice_64", kind="kdk", set="lattice", n=64 ** 3, box=1.0, rs_cells=0.625, theta=0.5,
             ngrid=128),
    ]


def draw(rng):
    """One case of the same kinds and ranges, no larger than the listed ones."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["forces", "forces", "grad", "linear_loss", "forces64", "keys", "pm", "sph", "kdk"])
    kinds = {"forces": ["uniform", "lattice", "clustered", "zoom"], "grad": ["lattice", "clustered"],
             "linear_loss": ["lattice", "clustered"], "forces64": ["uniform", "lattice", "clustered"],
             "keys": ["uniform", "clustered", "zoom"], "pm": ["lattice", "clustered"],
             "sph": ["uniform", "lattice", "clustered"], "kdk": ["lattice", "uniform"]}
    top = {"forces": 3_000_000, "grad": 1_500_000, "linear_loss": 1_500_000, "forces64": 200_000,
           "keys": 16_000_000, "pm": 4_000_000, "sph": 1_500_000, "kdk": 600_000}
    c = dict(kind=kind, set=rng.choice(kinds[kind]), n=size(1000, top[kind]),
             box=rng.choice([1.0, 1.0, 2.0, 50.0, round(rng.uniform(0.5, 300.0), 3)]))
    if kind == "forces" and c["set"] == "zoom":
        c["n"] = size(1000, 400_000)   # thousands of interactions a particle
    if c["set"] == "lattice":
        c["n"] = max(10, round(c["n"] ** (1 / 3))) ** 3
    side = c["n"] ** (1 / 3)
    if kind in ("forces", "grad", "linear_loss", "forces64", "kdk"):
        c["rs_cells"] = rng.choice([0.625, 0.625, 0.8])
        c["theta"] = rng.choice([0.4, 0.5, 0.5, 0.6, 0.7])
    if kind in ("pm", "kdk"):
        c["ngrid"] = max(16, min(384, round(side * rng.uniform(1.0, 2.0))))
    if kind == "sph":
        c["n_ngb"] = rng.choice([16, 32, 48, 64, 100])
    return c


# ---------------------------------------------------------------- particle sets

def _device():
    return torch.device("cuda:0" if torch.cuda.is_available() else "cpu")


class _Draw:
    """Random numbers on the device from one seed."""

    def __init__(self, seed):
        self.dev = _device()
        self.g = torch.Generator(device=self.dev).manual_seed(int(seed))

    def rand(self, *shape):
        return torch.rand(*shape, dtype=torch.float64, device=self.dev, generator=self.g)

    def randn(self, *shape):
        return torch.randn(*shape, dtype=torch.float64, device=self.dev, generator=self.g)

    def perm(self, n):
        return torch.randperm(n, device=self.dev, generator=self.g)


def _lattice(d, n):
    """A cubic lattice and a Zel'dovich displacement from P(k) ~ k^-2, rms half a cell."""
    s = round(n ** (1 / 3))
    k = torch.fft.fftfreq(s, 1.0 / s, dtype=torch.float64, device=d.dev)
    kz = torch.fft.rfftfreq(s, 1.0 / s, dtype=torch.float64, device=d.dev)
    K = torch.meshgrid(k, k, kz, indexing="ij")
    k2 = K[0] ** 2 + K[1] ** 2 + K[2] ** 2
    keep = (k2 > 0) & (K[0].abs() < s // 2) & (K[1].abs() < s // 2) & (K[2].abs() < s // 2)
    amp = torch.where(keep, k2.clamp(min=1.0) ** -1.5, torch.zeros_like(k2))
    white = torch.fft.rfftn(d.randn(s, s, s))
    psi = torch.stack([torch.fft.irfftn(1j * Ka * amp * white, s=(s, s, s)) for Ka in K], -1).reshape(-1, 3)
    psi *= 0.5 / s / psi.square().sum(1).mean().sqrt()
    g = (torch.arange(s, dtype=torch.float64, device=d.dev) + 0.5) / s
    q = torch.stack(torch.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
    return q, psi


def _nfw_radius(d, conc):
    """r / r200 of an NFW profile cut at r200, one per entry of conc: inverse CDF by bisection in ln x."""
    def mu(x):
        return torch.log1p(x) - x / (1.0 + x)

    want = d.rand(conc.shape[0]) * mu(conc)
    lo, hi = torch.full_like(conc, math.log(1e-9)), conc.log()
    for _ in range(40):
        mid = 0.5 * (lo + hi)
        below = mu(mid.exp()) < want
        lo, hi = torch.where(below, mid, lo), torch.where(below, hi, mid)
    return (0.5 * (lo + hi)).exp() / conc


def _direction(d, n):
    v = d.randn(n, 3)
    return v / v.norm(dim=1, keepdim=True)


def _clustered(d, n, halos=2000):
    """60 % of the particles in NFW haloes with dN/dM ~ M^-1.9, the rest uniform, in random order."""
    a = -0.9
    m = (1e-5 ** a + d.rand(halos) * (1e-2 ** a - 1e-5 ** a)) ** (1.0 / a)
    m *= 0.6 / m.sum()
    n_halo = int(round(0.6 * n))
    edges = (m.cumsum(0) / 0.6 * n_halo).round().long().clamp(max=n_halo)
    edges[-1] = n_halo
    of = torch.searchsorted(edges, torch.arange(n_halo, device=d.dev), right=True)
    r200 = (3.0 * m / (800.0 * math.pi)) ** (1.0 / 3.0)
    conc = 5.0 + 10.0 * d.rand(halos)
    centre = d.rand(halos, 3)
    x = centre[of] + (r200[of] * _nfw_radius(d, conc[of]))[:, None] * _direction(d, n_halo)
    return torch.cat([x, d.rand(n - n_halo, 3)])[d.perm(n)]


def _particles(case, seed):
    """pos, displacement from the undisplaced set (lattice only), mass, eps, all FP64, in the case's box."""
    d = _Draw(seed)
    n, box = case["n"], case["box"]
    side = n ** (1 / 3)
    disp = None
    mass = torch.full((n,), 1.0 / n, dtype=torch.float64, device=d.dev)
    eps = torch.full((n,), box / (30.0 * side), dtype=torch.float64, device=d.dev)
    if case["set"] == "uniform":
        x = d.rand(n, 3)
    elif case["set"] == "lattice":
        x, disp = _lattice(d, n)
        disp = disp * box
    elif case["set"] == "clustered":
        x = _clustered(d, n)
    else:  # zoom: four fifths of the particles light, in an NFW sphere at the centre; the others 64 times heavier
        hr = n - n // 5
        conc = torch.full((hr,), 10.0, dtype=torch.float64, device=d.dev)
        x = torch.cat([0.5 + 0.1 * _nfw_radius(d, conc)[:, None] * _direction(d, hr), d.rand(n - hr, 3)])
        m = 1.0 / (hr + 64.0 * (n - hr))
        mass[:hr], mass[hr:] = m, 64.0 * m
        eps[:hr] *= 0.25
        p = d.perm(n)
        x, mass, eps = x[p], mass[p].contiguous(), eps[p].contiguous()
    pos = torch.remainder(x, 1.0) * box
    pos = torch.where(pos >= box, torch.zeros_like(pos), pos).contiguous()
    return pos, disp, mass, eps


def _inputs(case, seed):
    """Everything a pass starts from, as both run() and exact() take it."""
    pos, disp, mass, eps = _particles(case, seed)
    d = _Draw(seed + 1_000_003)
    n, box = case["n"], case["box"]
    s = dict(case=case, pos=pos, mass=mass, eps=eps, box=box)
    if "rs_cells" in case:
        s["r_s"] = case["rs_cells"] * box / n ** (1 / 3)
    if case["kind"] in ("grad", "linear_loss"):
        # the parameters of a fit, in torch's usual type: displacements from a known set, and masses
        disp = d.randn(n, 3) * (0.1 * box / n ** (1 / 3)) if disp is None else disp
        s["disp"] = disp.float().requires_grad_(True)
        s["mass32"] = mass.float().requires_grad_(True)
        s["w"] = d.randn(n, 3).float()
    elif case["kind"] == "kdk":
        omega = math.sqrt(4.0 * math.pi / box ** 3)  # total mass 1: the box's own dynamical time
        if disp is None:
            s["vel"] = omega * 0.5 * box / n ** (1 / 3) * d.randn(n, 3)
        else:
            s["pos"] = pos + disp
            s["vel"] = (omega * disp).contiguous()
        s["dt"] = 2e-3 / omega
    elif disp is not None:
        s["pos"] = pos + disp
    return s


# ---------------------------------------------------------------- one pass

def prepare(case, seed):
    s = _inputs(case, seed)
    if case["kind"] == "pm":
        s["plan"] = og.PMPlan(case["ngrid"])
        s["r_s"] = 1.25 * case["box"] / case["ngrid"]
    elif case["kind"] == "kdk":
        s["stepper"] = og.TreePMStepper(s["pos"], s["vel"], s["mass"], s["eps"], s["box"], s["r_s"], case["theta"],
                                        case["ngrid"])
    return s


def _tree(s):
    keys, order = og.keys_sort(s["pos"], s["box"], check=False)
    return og.tree_build(keys, order, s["pos"], s["mass"], s["eps"], s["box"], check=False)


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "forces":
        acc, total, _ = og.shortrange_accel(_tree(s), s["r_s"], case["theta"], check=False)
        return acc, total
    if kind == "forces64":
        acc, total, counts = og.shortrange_accel(_tree(s), s["r_s"], case["theta"], prec="fp64", counts=True,
                                                 check=False)
        return acc, total, counts
    if kind == "grad":
        acc = og.ShortRangeAccel.apply(s["pos"] + s["disp"].double(), s["mass32"].double(), s["eps"], s["box"],
                                       s["r_s"], case["theta"])
        return (acc.detach(), *torch.autograd.grad(acc, (s["disp"], s["mass32"]), s["w"]))
    if kind == "linear_loss":
        w = s["w"].detach().requires_grad_(True)
        loss = og.ShortRangeLinearLoss.apply(s["pos"] + s["disp"].double(), s["mass32"].double(), s["eps"], w,
                                             s["box"], s["r_s"], case["theta"])
        return (loss.detach().float(), *torch.autograd.grad(loss, (s["disp"], s["mass32"], w)))
    if kind == "keys":
        return og.keys_sort(s["pos"], s["box"], check=False)
    if kind == "pm":
        return og.pm_accel(s["plan"], s["pos"], s["mass"], s["box"], s["r_s"], check=False)
    if kind == "sph":
        return og.sph_density(_tree(s), case["n_ngb"], check=False)
    s["stepper"].step(s["dt"])
    return s["stepper"].pos, s["stepper"].vel, s["stepper"].acc_s, s["stepper"].acc_l


def _terms_per_particle(case):
    """Interactions a particle has, counted on sets of these kinds, within a factor of two."""
    cells = (case["rs_cells"] / 0.625) ** 3
    if case["set"] == "zoom":
        return 5100.0 * cells * math.sqrt(case["n"] / 187_501)
    if case["set"] == "clustered":
        return 300.0 * cells * math.sqrt(case["n"] / 64 ** 3)
    return 88.0 * cells


def work(case):
    n, kind = case["n"], case["kind"]
    inputs, acc = 40, 12   # position, mass, softening; an FP32 acceleration
    if kind == "forces":
        return {"bytes": n * (inputs + acc), "flops": 45.0 * n * _terms_per_particle(case)}
    if kind == "forces64":
        return {"bytes": n * (inputs + 28), "flops": 45.0 * n * _terms_per_particle(case)}
    if kind in ("grad", "linear_loss"):  # displacement, float mass, weights in; gradients out
        both = 45 + 70 if kind == "grad" else 80  # two walks, or one for both
        return {"bytes": n * (inputs + 24 + acc + 16), "flops": both * n * _terms_per_particle(case)}
    if kind == "keys":
        return {"bytes": n * 36, "flops": 0}
    if kind == "sph":  # at least one evaluation of every neighbour
        return {"bytes": n * (inputs + 20), "flops": 25.0 * n * case["n_ngb"]}
    mesh = 2 * 2.5 * case["ngrid"] ** 3 * 3 * math.log2(case["ngrid"])  # a real transform each way
    if kind == "pm":
        return {"bytes": n * (32 + acc), "flops": mesh + 300.0 * n}
    # kdk: position and velocity in and out, mass, softening, both accelerations in and out
    return {"bytes": n * (4 * 24 + 16 + 4 * acc), "flops": mesh + n * (300.0 + 45.0 * _terms_per_particle(case))}


# ---------------------------------------------------------------- the method in FP64

def _wrap(pos, box):
    return pos - box * torch.floor(pos / box)


def _image(t, box):
    """Minimum image of a difference."""
    t = torch.where(t > 0.5 * box, t - box, t)
    return torch.where(t < -0.5 * box, t + box, t)


def _spread(v):
    out = torch.zeros_like(v)
    for b in range(21):
        out |= ((v >> b) & 1) << (3 * b)
    return out


class _Octree:
    """Cells of the 21-level grid with more than LEAF members are split; particles in Morton order."""

    def __init__(self, pos, mass, h, box):
        self.box = box
        x = _wrap(pos, box)
        cell = torch.floor((x / box) * 2.0 ** 21).long().clamp(0, 2 ** 21 - 1)
        key = (_spread(cell[:, 0]) << 2) | (_spread(cell[:, 1]) << 1) | _spread(cell[:, 2])
        key, self.order = torch.sort(key, stable=True)
        self.x, self.m, self.h, cell = x[self.order], mass[self.order], h[self.order], cell[self.order]
        dev, n = pos.device, pos.shape[0]
        self.n = n
        cols = {k: [] for k in ("first", "count", "level", "parent", "child", "nchild", "m", "mx", "h", "c")}
        live = torch.arange(n, device=dev)            # particles in cells of the current level
        owner = torch.zeros(n, dtype=torch.long, device=dev)   # the node one level up
        self.leaf_of = torch.zeros(n, dtype=torch.long, device=dev)
        base, last = 0, None
        for lev in range(22):
            pre = key[live] >> (63 - 3 * lev)
            new = torch.ones_like(pre, dtype=torch.bool)
            new[1:] = pre[1:] != pre[:-1]
            start = new.nonzero()[:, 0]
            of = new.long().cumsum(0) - 1
            cnt = torch.diff(start, append=torch.tensor([live.shape[0]], device=dev))
            k = start.shape[0]
            sums = [torch.zeros(k, dtype=torch.float64, device=dev).index_add_(0, of, self.m[live]),
                    torch.zeros(k, 3, dtype=torch.float64, device=dev).index_add_(
                        0, of, self.m[live][:, None] * self.x[live])]
            hmax = torch.zeros(k, dtype=torch.float64, device=dev).scatter_reduce_(0, of, self.h[live], "amax")
            side = box * 2.0 ** -lev
            cen = ((cell[live[start]] >> (21 - lev)).double() + 0.5) * side
            parent = owner[live[start]] if lev else torch.full((1,), -1, dtype=torch.long, device=dev)
            if lev:  # children of one node are consecutive
                nch = torch.bincount(parent - last, minlength=self._k)
                first_child = base + nch.cumsum(0) - nch
                cols["child"].append(first_child)
                cols["nchild"].append(nch)
            split = (cnt > LEAF) & (lev < 21)
            for name, v in (("first", live[start]), ("count", cnt), ("level", torch.full_like(cnt, lev)),
                            ("parent", parent), ("m", sums[0]), ("mx", sums[1]), ("h", hmax), ("c", cen)):
                cols[name].append(v)
            self.leaf_of[live] = base + of
            owner[live] = base + of
            last, self._k = base, k
            base += k
            live = live[split[of]]
            if live.shape[0] == 0:
                break
        cols["child"].append(torch.zeros(self._k, dtype=torch.long, device=dev))
        cols["nchild"].append(torch.zeros(self._k, dtype=torch.long, device=dev))
        for name, v in cols.items():
            setattr(self, "n" + name, torch.cat(v))
        self.ncom = self.nmx / self.nm[:, None]
        self.nside = box * 2.0 ** -self.nlevel.double()


def _expand(of, first, count):
    """(of repeated count times, first + 0, 1, ...) for ragged ranges."""
    i = torch.repeat_interleave(torch.arange(of.shape[0], device=of.device), count)
    start = count.cumsum(0) - count
    return of[i], first[i] + torch.arange(i.shape[0], device=of.device) - start[i]


def _frontier(tree, targets, decide):
    """Breadth-first over (target, node): decide(t, node) gives (accept, open); yields accepted (t, node) and (t, particle)."""
    t, node = targets, torch.zeros_like(targets)
    while t.shape[0]:
        accept, opened = decide(t, node)
        leaf = tree.nnchild[node] == 0
        pt, pj = _expand(t[opened & leaf], tree.nfirst[node[opened & leaf]], tree.ncount[node[opened & leaf]])
        yield t[accept], node[accept], pt, pj
        go = opened & ~leaf
        t, node = _expand(t[go], tree.nchild[node[go]], tree.nnchild[node[go]])


def _factor(r, h, r_s):
    """K_h(r) f(r) and its derivative over r."""
    v = (r / h).clamp(min=1e-300)
    rr = torch.where(r > 0, r, torch.ones_like(r))
    K, Kp = rr ** -3, -3.0 * rr ** -5
    h3 = h ** -3
    inner, mid = v < 0.5, (v >= 0.5) & (v < 1.0)
    K = torch.where(inner, h3 * (32.0 / 3.0 + v * v * (32.0 * v - 38.4)), K)
    Kp = torch.where(inner, h3 / h ** 2 * (96.0 * v - 76.8), Kp)
    K = torch.where(mid, h3 * (64.0 / 3.0 - 48.0 * v + 38.4 * v ** 2 - 32.0 / 3.0 * v ** 3 - 1.0 / (15.0 * v ** 3)), K)
    Kp = torch.where(mid, h3 / h ** 2 * (-48.0 / v + 76.8 - 32.0 * v + 0.2 / v ** 5), Kp)
    u = r / (2.0 * r_s)
    e = torch.exp(-u * u)
    f = torch.erfc(u) + 2.0 / math.sqrt(math.pi) * u * e
    fp = -r * e / (2.0 * math.sqrt(math.pi) * r_s ** 3)
    return K * f, Kp * f + K * fp


def _chunks(n, size):
    return (range(a, min(n, a + size)) for a in range(0, n, size))


def _walk(tree, r_s, theta, w=None):
    """Accelerations in tree order; with weights also dL/dx and dL/dm of L = sum w . a, the decisions held."""
    box, rc2, n, dev = tree.box, (RCUT * r_s) ** 2, tree.n, tree.x.device
    acc = torch.zeros(n, 3, dtype=torch.float64, device=dev)
    if w is not None:
        dx, gp, sp = torch.zeros_like(acc), torch.zeros_like(acc), torch.zeros_like(tree.m)
        gn, sn = torch.zeros_like(tree.ncom), torch.zeros_like(tree.nm)

    def decide(t, node):
        side = tree.nside[node]
        dc = _image(tree.x[t] - tree.nc[node], box).abs()
        near2 = (dc - 0.5 * side[:, None]).clamp(min=0.0).square().sum(1)
        far2 = (dc + 0.5 * side[:, None]).square().sum(1)
        d2 = _image(tree.x[t] - tree.ncom[node], box).square().sum(1)
        ok = (side * side < theta * theta * d2) & (dc.amax(1) > 0.6 * side) & (far2 < rc2)
        keep = near2 <= rc2
        return keep & ok & (d2 < rc2), keep & ~ok

    def add(t, xs, ms, hs, gs, ss, at):
        d = _image(tree.x[t] - xs, box)
        r = d.square().sum(1).sqrt()
        F, Fr = _factor(r, torch.maximum(tree.h[t], hs), r_s)
        acc.index_add_(0, t, (-ms * F)[:, None] * d)
        if w is not None:
            dw = (d * w[t]).sum(1)
            j = -(F[:, None] * w[t] + (Fr * dw)[:, None] * d)
            dx.index_add_(0, t, ms[:, None] * j)
            gs.index_add_(0, at, j)
            ss.index_add_(0, at, -F * dw)

    for part in _chunks(n, 8192):
        targets = torch.arange(part.start, part.stop, device=dev)
        for t, node, pt, pj in _frontier(tree, targets, decide):
            add(t, tree.ncom[node], tree.nm[node], tree.nh[node], *((gn, sn) if w is not None else (None, None)), node)
            inside = (_image(tree.x[pt] - tree.x[pj], box).square().sum(1) < rc2) & (pt != pj)
            pt, pj = pt[inside], pj[inside]
            add(pt, tree.x[pj], tree.m[pj], tree.h[pj], *((gp, sp) if w is not None else (None, None)), pj)
    if w is None:
        return acc, None, None
    # a node's centre of mass moves with its members: carry the node sums down to the leaves
    sn = sn + (gn * tree.ncom).sum(1)
    for lev in range(1, 22):
        k = (tree.nlevel == lev).nonzero()[:, 0]
        gn[k] += gn[tree.nparent[k]]
        sn[k] += sn[tree.nparent[k]]
    g = gn[tree.leaf_of]
    return acc, dx - tree.m[:, None] * (gp + g), sp + sn[tree.leaf_of] - (g * tree.x).sum(1)


def _unsort(tree, *values):
    out = []
    for v in values:
        o = torch.empty_like(v)
        o[tree.order] = v
        out.append(o)
    return out


def _kernel(q):
    u, v = (1.0 - q).clamp(min=0.0), (0.5 - q).clamp(min=0.0)
    return 2.0 * u ** 3 - 8.0 * v ** 3


def _sph(tree, n_ngb):
    """h with (32 / 3) sum w(r / h) = n_ngb by bisection, and the density at it, in tree order."""
    n, box, dev = tree.n, tree.box, tree.x.device
    hs, rho = torch.empty_like(tree.m), torch.empty_like(tree.m)
    up = tree.leaf_of.clone()
    for _ in range(22):
        up = torch.where((tree.ncount[up] < n_ngb) & (tree.nparent[up] >= 0), tree.nparent[up], up)
    guess = 1.3 * tree.nside[up] * (3.0 * n_ngb / (4.0 * math.pi * tree.ncount[up].double())) ** (1.0 / 3.0)
    for part in _chunks(n, 16384):
        todo = torch.arange(part.start, part.stop, device=dev)
        R = guess[todo].clamp(max=0.5 * box)
        while todo.shape[0]:
            reach = torch.zeros_like(tree.m)
            reach[todo] = R

            def decide(t, node):
                dc = _image(tree.x[t] - tree.nc[node], box).abs() - 0.5 * tree.nside[node][:, None]
                near = dc.clamp(min=0.0).square().sum(1) <= reach[t] ** 2
                return torch.zeros_like(near), near

            ts, rs, js = [], [], []
            for _, _, pt, pj in _frontier(tree, todo, decide):
                r = _image(tree.x[pt] - tree.x[pj], box).square().sum(1).sqrt()
                near = r < reach[pt]
                ts.append(pt[near])
                rs.append(r[near])
                js.append(pj[near])
            t, r, j = torch.cat(ts) - part.start, torch.cat(rs), torch.cat(js)
            size = part.stop - part.start

            def total(hh, weight=None):
                v = _kernel(r / hh[t])
                return torch.zeros(size, dtype=torch.float64, device=dev).index_add_(
                    0, t, v if weight is None else v * weight)

            local = todo - part.start
            hi = torch.full((size,), box, dtype=torch.float64, device=dev)
            hi[local] = R
            enough = ((32.0 / 3.0) * total(hi))[local] >= n_ngb
            lo = 0.3 * hi
            while bool(((32.0 / 3.0) * total(lo) > n_ngb)[local][enough].any()):
                lo = torch.where((32.0 / 3.0) * total(lo) > n_ngb, 0.5 * lo, lo)
            for _ in range(52):
                mid = 0.5 * (lo + hi)
                below = (32.0 / 3.0) * total(mid) < n_ngb
                lo, hi = torch.where(below, mid, lo), torch.where(below, hi, mid)
            done = todo[enough]
            hh = 0.5 * (lo + hi)
            hs[done] = hh[local][enough]
            rho[done] = (8.0 / math.pi * total(hh, tree.m[j]) / hh ** 3)[local][enough]
            todo, R = todo[~enough], 1.5 * R[~enough]
    return hs, rho


def _mesh(pos, mass, box, N, r_s):
    """Long-range accelerations: CIC, the Green's function with both windows divided out, four-point differences."""
    dev = pos.device
    u = _wrap(pos, box) * N / box
    i0 = torch.floor(u)
    f, i0 = u - i0, i0.long() % N
    corners = [(a, b, c) for a in (0, 1) for b in (0, 1) for c in (0, 1)]

    def at(o):
        i = [(i0[:, a] + o[a]) % N for a in range(3)]
        wt = [f[:, a] if o[a] else 1.0 - f[:, a] for a in range(3)]
        return (i[0] * N + i[1]) * N + i[2], wt[0] * wt[1] * wt[2]

    rho = torch.zeros(N ** 3, dtype=torch.float64, device=dev)
    for o in corners:
        i, wt = at(o)
        rho.index_add_(0, i, mass * wt)
    k = torch.fft.fftfreq(N, 1.0 / N, dtype=torch.float64, device=dev)
    kz = torch.fft.rfftfreq(N, 1.0 / N, dtype=torch.float64, device=dev)
    K = torch.meshgrid(k, k, kz, indexing="ij")
    k2 = (2.0 * math.pi / box) ** 2 * (K[0] ** 2 + K[1] ** 2 + K[2] ** 2)
    S = (torch.sinc(K[0] / N) * torch.sinc(K[1] / N) * torch.sinc(K[2] / N)) ** 4
    k2[0, 0, 0] = 1.0
    green = -4.0 * math.pi * torch.exp(-k2 * r_s ** 2) / (k2 * S) / (box / N) ** 3
    green[0, 0, 0] = 0.0
    phi = torch.fft.irfftn(torch.fft.rfftn(rho.view(N, N, N)) * green, s=(N, N, N))
    acc = torch.zeros_like(pos)
    for a in range(3):
        p = [torch.roll(phi, -s, a) for s in (-2, -1, 1, 2)]
        F = (-((2.0 / 3.0) * (p[2] - p[1]) - (1.0 / 12.0) * (p[3] - p[0])) * (N / box)).reshape(-1)
        for o in corners:
            i, wt = at(o)
            acc[:, a] += wt * F[i]
    return acc


def exact(case, seed):
    kind = case["kind"]
    if kind == "keys" or (kind == "forces" and case["n"] > 4_000_000):
        return None  # whole numbers; more than 10^10 interactions
    s = _inputs(case, seed)
    pos, mass, box = s["pos"], s["mass"], s["box"]
    if kind == "pm":
        return _mesh(pos, mass, box, case["ngrid"], 1.25 * box / case["ngrid"])
    if kind in ("grad", "linear_loss"):
        pos, mass = pos + s["disp"].detach().double(), s["mass32"].detach().double()

    def tree():
        return _Octree(pos, mass, 2.8 * s["eps"], box)

    if kind == "sph":
        T = tree()
        return (*_unsort(T, *_sph(T, case["n_ngb"])), None)
    if kind in ("forces", "forces64"):
        T = tree()
        acc, = _unsort(T, _walk(T, s["r_s"], case["theta"])[0])
        return (acc, None) if kind == "forces" else (acc, None, None)
    if kind in ("grad", "linear_loss"):
        T = tree()
        w = s["w"].double()
        acc, dx, dm = _unsort(T, *_walk(T, s["r_s"], case["theta"], w[T.order]))
        return (acc, dx, dm) if kind == "grad" else ((acc * w).sum(), dx, dm, acc)

    def forces():
        T = tree()
        return (*_unsort(T, _walk(T, s["r_s"], case["theta"])[0]), _mesh(pos, mass, box, case["ngrid"], s["r_s"]))

    short, long = forces()
    vel = s["vel"] + 0.5 * s["dt"] * (short + long)
    pos = pos + s["dt"] * vel
    short, long = forces()
    return pos, vel + 0.5 * s["dt"] * (short + long), short, long
