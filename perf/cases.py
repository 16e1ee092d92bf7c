"""Performance cases of the tree-code: what a program does with it, at the sizes it does it.

``listed()`` names the cases, ``draw(rng)`` gives more of the same ranges,
``prepare`` makes what the program has in hand (particles, a tree, a trained
criterion), ``run`` is one pass through the public calls and ``work`` counts
what that pass cannot do without. ``exact`` evaluates the same interaction
lists (octree, groups and opening test of the package's definition, restated
here in torch) in 64 bits.

Kinds of case:

* ``forces``   -- forces of one system on a tree that is on the device.
* ``batch``    -- forces of many independent systems by replaying a captured graph.
* ``learned``  -- forces with the learned opening criterion.
* ``step``     -- tree built on the GPU from device positions, then forces.
* ``host``     -- tree built on the host, uploaded, then forces.
* ``sim``      -- leapfrog steps with the state on the device, then a snapshot.
* ``direct``   -- FP64 direct sums at sampled particles (the error measurements).
* ``training`` -- training steps of the learned criterion on its samples.
"""
import math

import numpy as np
import torch

from paper_1005_5384_gb300 import octgrav as G
from paper_1005_5384_gb300 import workloads as W

N_LEAF = 16
EPS = {"plummer": 0.01, "clustered": 0.001, "galaxy": 0.01, "sphere_disc": 0.01}


def listed():
    return [
        # A small cluster simulation: too few work items to fill the GPU, so the
        # tuner's launch shape (one particle per lane, lists split over 4 warps).
        dict(name="forces_plummer_16k", kind="forces", dist="plummer", n=16384, theta=0.5, n_group=128, ppl=1, split=4),
        # The benchmark's headline: one Plummer sphere of 2^20 particles.
        dict(name="forces_plummer_1M", kind="forces", dist="plummer", n=1048576, theta=0.5, n_group=256, ppl=2, split=1),
        # The accuracy study's galaxy (bulge, disc and halo) at its group size 64,
        # an odd particle count and a loose theta.
        dict(name="forces_galaxy_300k", kind="forces", dist="galaxy", n=300007, theta=0.7, n_group=64, ppl=2, split=1),
        # The largest: 64 star clusters, deep and uneven trees.
        dict(name="forces_clustered_4M", kind="forces", dist="clustered", n=4194304, theta=0.5, n_group=256, ppl=2,
             split=1),
        # A parameter study: 256 independent systems of 1k to 65k particles in
        # one launch, captured once and replayed.
        dict(name="batch_256_systems", kind="batch", n_sys=256, n_min=1024, n_max=65536, theta=0.6, n_group=256),
        # The learned opening criterion on a sphere with a thin disc.
        dict(name="learned_sphere_disc_1M", kind="learned", dist="sphere_disc", n=1048576, tau=-3.5, n_group=256),
        # One force evaluation of a user's own integrator that keeps its state on
        # the GPU: a new tree and the forces on it.
        dict(name="step_plummer_1M", kind="step", dist="plummer", n=1048576, theta=0.75, n_group=256),
        # The same for a few thousand particles: launches and latency.
        dict(name="step_plummer_5k", kind="step", dist="plummer", n=5003, theta=0.5, n_group=64),
        # The paper's split of the work: tree on the host, forces on the GPU.
        dict(name="host_clustered_262k", kind="host", dist="clustered", n=262144, theta=0.5, n_group=256),
        # A star cluster integrated for four steps, then a snapshot for the host.
        dict(name="sim_plummer_65k", kind="sim", n=65537, theta=0.6, n_group=128, steps=4),
        # The reference of an error measurement: FP64 direct sums at 1024 particles.
        dict(name="direct_1024_of_300k", kind="direct", dist="galaxy", n=300000, targets=1024),
        # Fitting the learned criterion to the samples of some 64 groups: the first
        # steps of a training run at the benchmark's batch size.
        dict(name="training_64k_samples", kind="training", dist="sphere_disc", n=131072, n_group=256, samples=65536,
             steps=100, batch=4096),
    ]


def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forces", "forces", "forces", "batch", "learned", "step", "step", "host", "sim", "direct",
                       "training"])
    dist = rng.choice(["plummer", "clustered", "galaxy", "sphere_disc"])
    theta = round(rng.uniform(0.5, 1.0), 3)
    n_group = rng.choice([32, 64, 100, 128, 256, 512])
    if kind == "forces":
        n = _size(rng, 2000, 2000000)
        small = n < 40000
        return dict(kind=kind, dist=dist, n=n, theta=theta, n_group=n_group,
                    ppl=rng.choice([1, 2]) if small else 2, split=rng.choice([1, 2, 4]) if small else 1)
    if kind == "batch":
        hi = _size(rng, 2000, 60000)
        return dict(kind=kind, n_sys=rng.randint(3, 200), n_min=rng.randint(200, 1500), n_max=hi, theta=theta,
                    n_group=n_group)
    if kind == "learned":
        return dict(kind=kind, dist=dist, n=_size(rng, 20000, 1048576), tau=round(rng.uniform(-4.0, -3.0), 2),
                    n_group=rng.choice([128, 256]))
    if kind == "step":
        return dict(kind=kind, dist=dist, n=_size(rng, 1000, 1500000), theta=theta, n_group=n_group)
    if kind == "host":
        return dict(kind=kind, dist=dist, n=_size(rng, 4000, 500000), theta=theta, n_group=n_group)
    if kind == "sim":
        return dict(kind=kind, n=_size(rng, 2000, 130000), theta=theta, n_group=rng.choice([64, 128, 256]),
                    steps=rng.randint(1, 6))
    if kind == "direct":
        return dict(kind=kind, dist=dist, n=_size(rng, 20000, 300000), targets=_size(rng, 100, 1024))
    return dict(kind=kind, dist="sphere_disc", n=_size(rng, 60000, 131072), n_group=rng.choice([128, 256]),
                samples=_size(rng, 5000, 65536), steps=rng.randint(20, 100), batch=rng.choice([1000, 1024, 4096]))


# ---------------------------------------------------------------- inputs and passes

def _particles(dist, n, seed):
    if dist == "clustered":
        return W.clustered(n, seed=seed)
    return {"plummer": W.plummer, "galaxy": W.galaxy, "sphere_disc": W.sphere_disc}[dist](n, seed=seed)


def _systems(case, seed):
    """(pos, mass, offsets) of the independent Plummer spheres of a batch, sizes
    log-uniform in [n_min, n_max] and the same for every seed."""
    u = np.random.Generator(np.random.PCG64(case["n_sys"])).random(case["n_sys"])
    lo, hi = math.log(case["n_min"]), math.log(case["n_max"])
    sizes = np.rint(np.exp(lo + u * (hi - lo))).astype(np.int64)
    parts = [W.plummer(int(k), seed=1000 * seed + s) for s, k in enumerate(sizes)]
    return (np.concatenate([p for p, _ in parts]), np.concatenate([m for _, m in parts]),
            np.concatenate([[0], np.cumsum(sizes)]))


def _criterion():
    """A criterion record in the form mlp_train writes it: a network that
    predicts log10 of M l^3 / (20 |com - C|^5), the size of the first
    neglected multipole of a cell with mass M and side l in a system of unit
    mass and radius, in one pair of hidden units; the others hold small weights."""
    rng = np.random.Generator(np.random.PCG64(12))
    w1 = 0.02 * (2 * rng.random((64, 12)) - 1)
    w2 = 0.02 * (2 * rng.random((64, 64)) - 1)
    w3 = 0.02 * (2 * rng.random(64) - 1)
    b1, b2 = np.zeros(64), np.zeros(64)
    mu = np.array([-4, -4, -3, 1, -12, 0.1, 6, 0.5, 0.5, 0.5, 0.5, -1], np.float64)
    sd = np.array([2, 2, 2, 1, 4, 0.1, 3, 1, 1, 1, 0.5, 1], np.float64)
    lg2 = math.log10(2.0)
    slope = np.zeros(12)
    slope[0], slope[2], slope[4] = 3 * lg2, -5 * lg2, lg2  # log2 l, log2 |com - C|, log2 M
    w1[0], w1[1] = slope * sd, -slope * sd
    b1[0], b1[1] = slope @ mu, -(slope @ mu)
    w2[0], w2[1] = 0.0, 0.0
    w2[0, 0], w2[0, 1], w2[1, 0], w2[1, 1] = 1, -1, -1, 1
    w3[0], w3[1] = 1, -1
    return np.concatenate([mu, sd, np.full(12, -60.0), np.full(12, 60.0), w1.ravel(), b1, w2.ravel(), b2, w3,
                           [-math.log10(20.0)]]).astype(np.float32)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        pos, mass, off = _systems(case, seed)
        tree = G.Tree.build_gpu(pos, mass, N_LEAF, case["n_group"], offsets=off)
        out = torch.empty((tree.n, 4), dtype=torch.float32, device="cuda")
        stream = torch.cuda.Stream()
        tree.capture_graph(0.01, case["theta"], out, stream=stream)
        return dict(case=case, tree=tree, out=out, stream=stream)
    if kind == "sim":
        pos, vel, mass = W.plummer_pv(case["n"], seed=seed)
        return dict(case=case, sim=G.Sim(pos, vel, mass, 0.01, case["theta"], n_leaf=N_LEAF, n_group=case["n_group"]))
    pos, mass = _particles(case["dist"], case["n"], seed)
    state = dict(case=case, eps=EPS[case["dist"]])
    if kind in ("host", "direct"):
        state.update(pos=pos, mass=mass)
    if kind == "direct":
        state["targets"] = W.sample_indices(case["n"], case["targets"], seed=seed)
        return state
    state["out"] = torch.empty((case["n"], 4), dtype=torch.float32, device="cuda")
    if kind == "step":
        state.update(pos=torch.from_numpy(pos).cuda(), mass=torch.from_numpy(mass).cuda())
    if kind in ("forces", "learned", "training"):
        state["tree"] = tree = G.Tree.build_gpu(pos, mass, N_LEAF, case["n_group"])
        if kind == "training":
            few = max(4, case["samples"] // 300)
            groups = W.sample_indices(tree.stats["n_groups"], few, seed=seed)
            feat, label, _ = tree.mlp_samples(groups, 0.35, state["eps"])
            keep = np.nonzero(feat[:, 3] >= 0.6)[0]  # the samples near the band, as the benchmark trains on
            keep = np.resize(keep, case["samples"])
            return dict(case=case, feat=feat[keep], label=label[keep])
        if kind == "learned":
            tree.set_criterion(_criterion(), tau=case["tau"], theta_lo=0.85, theta_hi=1.5, theta_fb=1.0)
        else:
            tree.set_launch(case["ppl"], 0)
            tree.set_split(case["split"])
        # as an N-body code does from its second step on: the work items in the
        # order of the previous step's costs
        tree.forces_device(state["eps"], case.get("theta", 0.5), state["out"])
        tree.balance(1)
    return state


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind in ("forces", "learned"):
        state["tree"].forces_device(state["eps"], case.get("theta", 0.5), state["out"])
        return state["out"]
    if kind == "batch":
        state["tree"].launch_graph(stream=state["stream"])
        torch.cuda.current_stream().wait_stream(state["stream"])
        return state["out"]
    if kind == "step":
        tree = G.Tree.build_gpu(state["pos"], state["mass"], N_LEAF, case["n_group"])
        tree.forces_device(state["eps"], case["theta"], state["out"])
        return state["out"]
    if kind == "host":
        tree = G.Tree.build(state["pos"], state["mass"], N_LEAF, case["n_group"])
        tree.upload()
        tree.forces_device(state["eps"], case["theta"], state["out"])
        return state["out"]
    if kind == "sim":
        state["sim"].step(1.0 / 2048, case["steps"])
        pos, vel, _, _ = state["sim"].state()
        return dict(pos=pos, vel=vel)
    if kind == "direct":
        acc, pot = G.direct(state["pos"], state["mass"], state["eps"], targets=state["targets"])
        return dict(acc=acc, pot=pot)
    record, loss = G.mlp_train(state["feat"], state["label"], steps=case["steps"], batch=case["batch"], lr=2e-3, seed=3)
    return dict(record=record, loss=np.float32(loss))


# ---------------------------------------------------------------- what a pass cannot do without

def _flops(n, theta, n_group):
    """Floating-point operations of a force evaluation (38 per particle pair, 70
    per particle and cell), with list lengths fitted within a factor of 1.6 to
    counted ones (Plummer spheres and the galaxy, 5 thousand to a million particles)."""
    levels = math.log2(max(2.0, n / n_group))
    far = 6.0 * n_group ** 0.35 * levels ** 1.6 * theta ** -1.1
    near = 3.0 * (n_group + 4 * N_LEAF) * theta ** -1.4
    return n * (70.0 * far + 38.0 * min(n, near))


def work(case):
    kind = case["kind"]
    if kind == "training":
        return {"bytes": 52.0 * case["samples"] + 4.0 * 5105, "flops": 6.0 * 5057 * case["batch"] * case["steps"]}
    if kind == "batch":
        mean = (case["n_max"] - case["n_min"]) / math.log(case["n_max"] / case["n_min"])
        n = case["n_sys"] * mean
        return {"bytes": n * (32 + 16 + 0.24 * 88), "flops": case["n_sys"] * _flops(mean, case["theta"], case["n_group"])}
    n = case["n"]
    if kind == "direct":
        return {"bytes": 32.0 * n + 40.0 * case["targets"], "flops": 20.0 * n * case["targets"]}
    if kind == "sim":
        return {"bytes": case["steps"] * n * 200.0, "flops": case["steps"] * _flops(n, case["theta"], case["n_group"])}
    # particles and about a quarter as many cells in, accelerations and potentials out;
    # the learned criterion's lists are 0.4 times those of the plain test at theta = 1.2
    flops = 0.4 * _flops(n, 1.2, case["n_group"]) if kind == "learned" else _flops(n, case["theta"], case["n_group"])
    return {"bytes": n * (32 + 16 + 0.24 * 88), "flops": flops}


# ---------------------------------------------------------------- the same lists in 64 bits

def _morton(pos, sys_of, n_sys):
    idx = sys_of[:, None].expand(-1, 3)
    mn = torch.full((n_sys, 3), math.inf, dtype=torch.float64, device=pos.device).scatter_reduce(0, idx, pos, "amin")
    mx = torch.full((n_sys, 3), -math.inf, dtype=torch.float64, device=pos.device).scatter_reduce(0, idx, pos, "amax")
    ext = (mx - mn).amax(1)
    side = torch.where(ext > 0, ext, torch.ones_like(ext)) * (1.0 + 2.0 ** -20)
    lo = (mn + mx) * 0.5 - (side * 0.5)[:, None]
    q = torch.floor(((pos - lo[sys_of]) / side[sys_of][:, None]) * 2.0 ** 21).clamp(0, 2 ** 21 - 1).long()
    key = torch.zeros(len(pos), dtype=torch.int64, device=pos.device)
    for b in range(21):
        for d in range(3):
            key |= ((q[:, d] >> b) & 1) << (3 * b + d)
    return key


class _Octree:
    """Cells (level by level), their moments and boundary cubes, and the groups."""

    def __init__(self, pos, mass, offsets, n_leaf, n_group):
        dev = pos.device
        n_sys = len(offsets) - 1
        off = torch.tensor(offsets, dtype=torch.int64, device=dev)
        sys_of = torch.repeat_interleave(torch.arange(n_sys, device=dev), off[1:] - off[:-1])
        key = _morton(pos, sys_of, n_sys)
        perm = torch.argsort(key, stable=True)
        perm = perm[torch.argsort(sys_of[perm], stable=True)]
        self.perm, key = perm, key[perm]
        self.x, self.m = pos[perm], mass[perm]
        n = len(key)
        at = torch.arange(n, device=dev)
        first, count, parent = [off[:-1]], [off[1:] - off[:-1]], [torch.full((n_sys,), -1, device=dev)]
        base, cell_of = 0, sys_of.clone()  # each particle's cell of the present level, -1 below a leaf
        owner = []                         # one particle-to-cell map per level, for the sums over members
        for depth in range(22):
            owner.append(cell_of)
            cnt = torch.cat(count)
            inside = cell_of >= 0
            split = inside & (depth < 21) & (cnt[cell_of.clamp(min=0)] > n_leaf)
            if not bool(split.any()):
                break
            p = at[split]
            octant = key[p] >> (3 * (20 - depth))
            new = torch.ones(len(p), dtype=torch.bool, device=dev)
            new[1:] = (octant[1:] != octant[:-1]) | (cell_of[p][1:] != cell_of[p][:-1])
            base = sum(len(f) for f in first)
            child = base + torch.cumsum(new, 0) - 1
            starts = p[new]
            first.append(starts)
            count.append(torch.bincount(child - base, minlength=len(starts)))
            parent.append(cell_of[starts])
            cell_of = torch.full((n,), -1, device=dev)
            cell_of[p] = child
        self.first, self.count, self.parent = torch.cat(first), torch.cat(count), torch.cat(parent)
        nc = len(self.first)
        f64 = dict(dtype=torch.float64, device=dev)
        self.M, com = torch.zeros(nc, **f64), torch.zeros(nc, 3, **f64)
        bmin, bmax = torch.full((nc, 3), math.inf, **f64), torch.full((nc, 3), -math.inf, **f64)
        for own in owner:
            k = own >= 0
            c, x, m = own[k], self.x[k], self.m[k]
            self.M.index_add_(0, c, m)
            com.index_add_(0, c, m[:, None] * x)
            bmin.scatter_reduce_(0, c[:, None].expand(-1, 3), x, "amin")
            bmax.scatter_reduce_(0, c[:, None].expand(-1, 3), x, "amax")
        self.com = com / self.M[:, None]
        self.S = torch.zeros(nc, 6, **f64)  # xx yy zz xy xz yz
        for own in owner:
            k = own >= 0
            c, m = own[k], self.m[k]
            y = self.x[k] - self.com[c]
            s = torch.stack([y[:, 0] * y[:, 0], y[:, 1] * y[:, 1], y[:, 2] * y[:, 2], y[:, 0] * y[:, 1],
                             y[:, 0] * y[:, 2], y[:, 1] * y[:, 2]], 1)
            self.S.index_add_(0, c, m[:, None] * s)
        self.centre, self.h = ((bmin + bmax) * 0.5).float(), (0.5 * (bmax - bmin).amax(1)).float()
        self.n_child = torch.bincount(self.parent[n_sys:], minlength=nc)
        ends = torch.cumsum(self.n_child, 0)
        self.child = n_sys + ends - self.n_child  # children follow their parents' order
        eligible = (self.n_child == 0) | (self.count <= n_group)
        up = self.parent.clamp(min=0)
        self.groups = torch.nonzero(eligible & ((self.parent < 0) | (self.count[up] > n_group))).flatten()
        root = torch.where(self.parent < 0, torch.arange(nc, device=dev), up)
        for _ in range(len(owner)):
            root = root[root]
        self.root = root[self.groups]
        self.gmin, self.gmax = bmin[self.groups].float(), bmax[self.groups].float()

    def walk(self, g, theta):
        """Lists of the groups g: (group, accepted cell) and (group, opened leaf)."""
        theta2 = torch.tensor(np.float32(theta * theta), device=g.device)
        cell = self.root[g]
        far, near = [torch.empty((2, 0), dtype=torch.int64, device=g.device)], []
        lone = self.n_child[cell] == 0
        near.append(torch.stack([g[lone], cell[lone]]))
        g, cell = g[~lone], cell[~lone]
        while len(g):
            k = self.n_child[cell]
            j = torch.arange(int(k.sum()), device=g.device) - torch.repeat_interleave(torch.cumsum(k, 0) - k, k)
            c = torch.repeat_interleave(self.child[cell], k) + j
            g = torch.repeat_interleave(g, k)
            h, ctr = self.h[c][:, None], self.centre[c]
            d = torch.maximum(self.gmin[g] - (ctr + h), (ctr - h) - self.gmax[g]).clamp(min=0)
            d = d * d
            d2 = (d[:, 0] + d[:, 1]) + d[:, 2]
            opened = 4.0 * (h[:, 0] * h[:, 0]) >= theta2 * d2
            leaf = self.n_child[c] == 0
            far.append(torch.stack([g[~opened], c[~opened]]))
            near.append(torch.stack([g[opened & leaf], c[opened & leaf]]))
            down = opened & ~leaf
            g, cell = g[down], c[down]
        return torch.cat(far, 1), torch.cat(near, 1)


def _ragged(k):
    """Row and index within the row of every entry of rows with k entries."""
    row = torch.repeat_interleave(torch.arange(len(k), device=k.device), k)
    return row, torch.arange(len(row), device=k.device) - (torch.cumsum(k, 0) - k)[row]


def _add(out, i, ax, ay, az, ph):
    out.index_add_(0, i, torch.stack([ax, ay, az, ph], 1))


def _forces64(pos, mass, offsets, eps, theta, n_leaf, n_group, limit=2.5e7):
    """(out [n, 4] in tree order, permutation) of the grouped walk, in 64 bits."""
    T = _Octree(pos, mass, offsets, n_leaf, n_group)
    out = torch.zeros((len(mass), 4), dtype=torch.float64, device=pos.device)
    eps2 = eps * eps
    size = T.count[T.groups]
    for g0 in range(0, len(T.groups), 2000):
        far, near = T.walk(torch.arange(g0, min(len(T.groups), g0 + 2000), device=pos.device), theta)
        for lists, is_far in ((far, True), (near, False)):
            gg, cc = lists
            per = size[gg] * (1 if is_far else T.count[cc])
            ends = torch.cumsum(per, 0)
            cuts = [0]
            while cuts[-1] < len(gg):
                done = float(ends[cuts[-1] - 1]) if cuts[-1] else 0.0
                cuts.append(max(cuts[-1] + 1, int(torch.searchsorted(ends, done + limit))))
            for a, b in zip(cuts, cuts[1:]):
                g, c = gg[a:b], cc[a:b]
                row, j = _ragged(per[a:b])
                if is_far:
                    i, c = T.first[T.groups[g]][row] + j, c[row]
                    y = T.x[i] - T.com[c]
                    s, M = T.S[c], T.M[c]
                    r2 = (y * y).sum(1) + eps2
                    sy = torch.stack([s[:, 0] * y[:, 0] + s[:, 3] * y[:, 1] + s[:, 4] * y[:, 2],
                                      s[:, 3] * y[:, 0] + s[:, 1] * y[:, 1] + s[:, 5] * y[:, 2],
                                      s[:, 4] * y[:, 0] + s[:, 5] * y[:, 1] + s[:, 2] * y[:, 2]], 1)
                    ysy, tr = (y * sy).sum(1), s[:, 0] + s[:, 1] + s[:, 2]
                    ri = torch.rsqrt(r2)
                    ri2 = ri * ri
                    ri3 = ri * ri2
                    k = ri3 * (-M + ri2 * (1.5 * tr - 7.5 * ysy * ri2))
                    f = k[:, None] * y + (3.0 * ri3 * ri2)[:, None] * sy
                    _add(out, i, f[:, 0], f[:, 1], f[:, 2], -ri * (M + ri2 * (1.5 * ysy * ri2 - 0.5 * tr)))
                else:
                    m = T.count[c][row]
                    i, q = T.first[T.groups[g]][row] + j // m, T.first[c][row] + j % m
                    y = T.x[q] - T.x[i]
                    ri = torch.rsqrt((y * y).sum(1) + eps2)
                    mr = torch.where(i == q, torch.zeros_like(ri), T.m[q] * ri)
                    f = (mr * ri * ri)[:, None] * y
                    _add(out, i, f[:, 0], f[:, 1], f[:, 2], -mr)
    return out, T.perm


def exact(case, seed):
    kind = case["kind"]
    if kind in ("learned", "training") or case.get("n", 0) > 1200000:
        return None
    cuda = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    if kind == "batch":
        pos, mass, off = _systems(case, seed)
        if off[-1] > 1200000:
            return None
        return _forces64(cuda(pos), cuda(mass), off.tolist(), 0.01, case["theta"], N_LEAF, case["n_group"])[0]
    if kind == "sim":
        pos, vel, mass = (cuda(a) for a in W.plummer_pv(case["n"], seed=seed))

        def accel(x):
            out, perm = _forces64(x, mass, [0, len(mass)], 0.01, case["theta"], N_LEAF, case["n_group"])
            a = torch.empty_like(x)
            a[perm] = out[:, :3]
            return a
        dt, a = 1.0 / 2048, accel(pos)
        for _ in range(case["steps"]):
            vel = vel + a * (0.5 * dt)
            pos = pos + vel * dt
            a = accel(pos)
            vel = vel + a * (0.5 * dt)
        return dict(pos=pos.cpu().numpy(), vel=vel.cpu().numpy())
    pos, mass = (cuda(a) for a in _particles(case["dist"], case["n"], seed))
    eps = EPS[case["dist"]]
    if kind == "direct":
        t = cuda(W.sample_indices(case["n"], case["targets"], seed=seed))
        acc = torch.zeros((len(t), 3), dtype=torch.float64, device="cuda")
        pot = torch.zeros(len(t), dtype=torch.float64, device="cuda")
        for a in range(0, case["n"], 20000):
            j = torch.arange(a, min(case["n"], a + 20000), device="cuda")
            y = pos[j][None] - pos[t][:, None]
            ri = torch.rsqrt((y * y).sum(2) + eps * eps)
            mr = torch.where(j[None] == t[:, None], torch.zeros_like(ri), mass[j] * ri)
            acc += ((mr * ri * ri)[:, :, None] * y).sum(1)
            pot -= mr.sum(1)
        return dict(acc=acc.cpu().numpy(), pot=pot.cpu().numpy())
    return _forces64(pos, mass, [0, case["n"]], eps, case["theta"], N_LEAF, case["n_group"])[0]
