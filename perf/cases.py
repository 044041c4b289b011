"""Timed cases of the tree-force library, through its public entry points.

Each case is one kind of call ("op") on one seeded particle set:

  sort        fdps_morton_sort_noalloc: keys and stable sort of device positions
  force       psys.set, calcForceAllAndWriteBack, psys.get of acceleration and
              potential, with device tensors or page-locked host arrays
  step        one kick-drift-kick step and a read of the whole state
  run         several steps by fdps_run and a read of the whole state
  neighbours  the short-range mode: neighbour counts and SPH densities
  userlaw     the interaction lists and a run-time compiled user law over them
  direct      the direct-sum reference at sampled rows

Sizes and parameters are those of the repository's workload table and tests
(Plummer 2^14 and 2^20, Hernquist 2^24, the clump mixture, ensembles of
256..65536-particle clusters, odd sizes such as 3,000,017), inputs are drawn
on the GPU from the seed.  `exact` restates the documented readings (root
box, keys, octree, opening test, force law, neighbour rule) with plain torch
operations in 64 bits.
"""
import math

import numpy as np
import torch

import paper_1601_03138_gb300 as G

DEV = "cuda" if torch.cuda.is_available() else "cpu"
F64 = torch.float64
MAX_LEVEL = 21

# The most interactions that `exact` evaluates (a few seconds on the GPU).
EXACT_PAIRS = 7e9

# Softened gravity with monopole and quadrupole superparticles, as a user of
# the run-time compiled laws writes it.
LAW = """
struct Force {
    float ax, ay, az, pot;
    __device__ void clear() { ax = ay = az = pot = 0.f; }
};
struct Law {
    __device__ void operator()(const Epi& i, const Epj* j, int nj, Force& f) const {
        for (int k = 0; k < nj; ++k) {
            const float dx = j[k].x - i.x, dy = j[k].y - i.y, dz = j[k].z - i.z;
            const float ri = rsqrtf(dx * dx + dy * dy + dz * dz + i.eps2);
            const float mri = j[k].m * ri;
            const float mri3 = mri * ri * ri;
            f.ax += mri3 * dx;
            f.ay += mri3 * dy;
            f.az += mri3 * dz;
            f.pot -= mri;
        }
    }
    __device__ void operator()(const Epi& i, const Spj* j, int nj, Force& f) const {
        for (int k = 0; k < nj; ++k) {
            const Spj& s = j[k];
            const float rx = i.x - s.x, ry = i.y - s.y, rz = i.z - s.z;
            const float ri = rsqrtf(rx * rx + ry * ry + rz * rz + i.eps2);
            const float ri2 = ri * ri, ri3 = ri * ri2, ri5 = ri3 * ri2;
            const float qx = s.qxx * rx + s.qxy * ry + s.qxz * rz;
            const float qy = s.qxy * rx + s.qyy * ry + s.qyz * rz;
            const float qz = s.qxz * rx + s.qyz * ry + s.qzz * rz;
            const float rqr = rx * qx + ry * qy + rz * qz;
            const float c = s.m * ri3 + 2.5f * rqr * ri5 * ri2;
            f.ax += qx * ri5 - c * rx;
            f.ay += qy * ri5 - c * ry;
            f.az += qz * ri5 - c * rz;
            f.pot -= s.m * ri + 0.5f * rqr * ri5;
        }
    }
};
"""


def listed():
    return [
        # the smallest call: a real-time loop's key sort, launch latency only
        dict(name="sort-4099", op="sort", model="plummer", n=4099),
        # a small star cluster integrated over many steps: latency of a step
        dict(name="run-cluster-2001", op="run", model="plummer", n=2001, steps=16, dt=1.0 / 128, eps=1.0 / 64,
             theta=0.5, quad=False, n_leaf=8, n_grp=64),
        # one step of the workload table's Plummer 2^14 sphere
        dict(name="step-plummer-16k", op="step", model="plummer", n=16384, dt=1.0 / 128, eps=1.0 / 64,
             theta=0.5, quad=False, n_leaf=8, n_grp=64),
        # the table's Plummer 2^20 sphere with its own tree parameters, data
        # of a torch program on the device
        dict(name="force-plummer-1m", op="force", model="plummer", n=1 << 20, where="device", eps=1.0 / 64,
             theta=0.5, quad=True, n_leaf=16, n_grp=128, fp64=False),
        # a ragged size of the strongly clustered mixture, monopoles and a
        # wide opening angle
        dict(name="force-clumpy-3m-mono", op="force", model="clumpy", n=3000017, where="device", eps=0.002,
             theta=0.7, quad=False, n_leaf=8, n_grp=256, fp64=False),
        # an N-body program that keeps its particles in host memory
        dict(name="host-hernquist-4m", op="force", model="hernquist", n=1 << 22, where="host", eps=0.005,
             theta=0.5, quad=True, n_leaf=16, n_grp=256, fp64=False),
        # the benchmark workload at the parameters its autotuner picks
        dict(name="step-hernquist-16m", op="step", model="hernquist", n=1 << 24, dt=1.0 / 512, eps=0.005,
             theta=0.5, quad=True, n_leaf=16, n_grp=256),
        # an ensemble of independent clusters with the table's parameters
        dict(name="run-ensemble-256", op="run", model="ensemble", n=256, steps=2, dt=1.0 / 256, eps=0.0,
             theta=0.5, quad=False, n_leaf=8, n_grp=64),
        # the all-FP64 pipeline, for reference-quality forces
        dict(name="fp64-plummer-100k", op="force", model="plummer", n=100003, where="device", eps=1.0 / 64,
             theta=0.5, quad=True, n_leaf=16, n_grp=128, fp64=True),
        # SPH density with gather radii of about 310 neighbours
        dict(name="neighbours-i-1m", op="neighbours", model="cube", n=1 << 20, mode=G.FDPS_CUTOFF_I,
             n_leaf=8, n_grp=32),
        # a user's own interaction law over the library's lists
        dict(name="userlaw-hernquist-1m", op="userlaw", model="hernquist", n=1 << 20, eps=0.005,
             theta=0.5, quad=True, n_leaf=16, n_grp=256),
        # the accuracy diagnostics' reference: 4096 rows of the direct sum
        dict(name="direct-4096-of-1m", op="direct", model="hernquist", n=1 << 20, rows=4096, eps=0.005),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["sort", "run", "step", "force", "force", "fp64", "ensemble", "neighbours", "userlaw", "direct"])
    if op == "sort":
        return dict(op="sort", model=rng.choice(["plummer", "cube", "clumpy"]), n=_log_int(rng, 256, G.FDPS_NOALLOC_MAX_N))
    if op == "neighbours":
        return dict(op=op, model=rng.choice(["cube", "cube", "plummer"]), n=_log_int(rng, 10000, 1 << 20),
                    mode=rng.randrange(4), n_leaf=rng.choice([8, 16]), n_grp=rng.choice([32, 64]))
    model = rng.choice(["plummer", "hernquist", "clumpy"])
    eps = {"plummer": 1.0 / 64, "hernquist": 0.005, "clumpy": 0.002}[model]
    if op == "direct":
        return dict(op=op, model=model, n=_log_int(rng, 10000, 1 << 21), rows=_log_int(rng, 64, 4096), eps=eps)
    c = dict(eps=eps, theta=rng.choice([0.3, 0.4, 0.5, 0.6, 0.7]), quad=rng.random() < 0.5,
             n_leaf=rng.choice([8, 16]), n_grp=rng.choice([64, 128, 256]))
    if op == "run":
        return dict(op=op, model=model, n=_log_int(rng, 512, 200000), steps=rng.choice([2, 4, 8, 16]), dt=1.0 / 512, **c)
    if op == "ensemble":
        c.update(eps=0.0, theta=0.5)
        return dict(op="run", model="ensemble", n=_log_int(rng, 8, 256), steps=rng.choice([2, 3, 4]), dt=1.0 / 512, **c)
    if op == "step":
        return dict(op=op, model=model, n=_log_int(rng, 4096, 1 << 22), dt=1.0 / 512, **c)
    if op == "userlaw":
        return dict(op=op, model=model, n=_log_int(rng, 10000, 1 << 20), **c)
    if op == "fp64":
        c["theta"] = max(c["theta"], 0.5)
        return dict(op="force", model=model, n=_log_int(rng, 1000, 100003), where="device", fp64=True, **c)
    return dict(op="force", model=model, n=_log_int(rng, 4096, 1 << 22), where=rng.choice(["device", "host"]), fp64=False, **c)


# ------------------------------------------------------------------ inputs

def _uniform(gen, *shape):
    return torch.rand(*shape, generator=gen, dtype=F64, device=DEV)


def _directions(gen, n):
    z = 2.0 * _uniform(gen, n) - 1.0
    phi = 2.0 * math.pi * _uniform(gen, n)
    s = torch.sqrt((1.0 - z * z).clamp(min=0.0))
    return torch.stack([s * torch.cos(phi), s * torch.sin(phi), z], 1)


def _plummer(gen, n, mass=1.0, a=1.0):
    """Plummer spheres (Aarseth, Henon & Wielen 1974) cut at 22.8 scale radii;
    `mass` and `a` are numbers or one value per particle."""
    xmax = (22.8 ** 2 / (1.0 + 22.8 ** 2)) ** 1.5
    x = (xmax * _uniform(gen, n)).clamp(min=1e-12)
    r = 1.0 / torch.sqrt(x ** (-2.0 / 3.0) - 1.0)
    q = torch.linspace(0.0, 1.0, 4097, dtype=F64, device=DEV)
    cdf = torch.cumsum(q ** 2 * (1.0 - q ** 2) ** 3.5, 0)
    cdf = cdf / cdf[-1]
    u = _uniform(gen, n)
    k = torch.searchsorted(cdf, u).clamp(1, 4096)
    w = ((u - cdf[k - 1]) / (cdf[k] - cdf[k - 1]).clamp(min=1e-300)).clamp(0.0, 1.0)
    speed = (q[k - 1] + w * (q[k] - q[k - 1])) * math.sqrt(2.0) * (1.0 + r * r) ** -0.25
    scale = torch.sqrt(torch.as_tensor(mass / a, dtype=F64, device=DEV))
    return _directions(gen, n) * (a * r)[:, None], _directions(gen, n) * (scale * speed)[:, None]


def _hernquist(gen, n):
    """Hernquist (1990) halo cut at 100 scale radii, with Gaussian velocities
    of the local dispersion (the isotropic Jeans equation), below escape."""
    s = torch.sqrt((100.0 / 101.0) ** 2 * _uniform(gen, n))
    r = (s / (1.0 - s)).clamp(min=1e-7)
    lr = torch.linspace(math.log(1e-7), math.log(101.0), 4096, dtype=F64, device=DEV)
    rt = torch.exp(lr)
    # sigma^2 = (1 / rho) int_r^inf rho M / r^2 dr, rho ~ 1 / (r (1 + r)^3)
    f = 1.0 / (rt * (1.0 + rt) ** 5) * rt
    tail = torch.flip(torch.cumsum(torch.flip(f, [0]), 0), [0]) * (lr[1] - lr[0])
    sig2 = tail * rt * (1.0 + rt) ** 3
    k = torch.searchsorted(rt, r).clamp(1, 4095)
    sig = torch.sqrt(sig2[k])
    v = torch.randn(n, 3, generator=gen, dtype=F64, device=DEV) * sig[:, None]
    vesc = torch.sqrt(2.0 / (1.0 + r))
    v = v * torch.clamp(0.95 * vesc / v.norm(dim=1).clamp(min=1e-30), max=1.0)[:, None]
    return _directions(gen, n) * r[:, None], v


def _clumpy(gen, n):
    """1000 Plummer clumps of log-normal masses (four fifths of the mass) in
    the unit sphere and a uniform background at rest."""
    nc = int(round(0.8 * n))
    m = torch.exp(torch.randn(1000, generator=gen, dtype=F64, device=DEV))
    m = 0.8 * m / m.sum()
    rc = 0.01 + 0.04 * _uniform(gen, 1000)
    centre = _directions(gen, 1000) * (_uniform(gen, 1000) ** (1.0 / 3.0))[:, None]
    edges = torch.cumsum(m, 0) / 0.8
    k = torch.searchsorted(edges, _uniform(gen, nc)).clamp(max=999)
    k, _ = torch.sort(k)
    p, v = _plummer(gen, nc, m[k], rc[k])
    bg = _directions(gen, n - nc) * (_uniform(gen, n - nc) ** (1.0 / 3.0))[:, None]
    return torch.cat([p + centre[k], bg]), torch.cat([v, torch.zeros_like(bg)])


def _inputs(case, seed):
    """pos, vel, mass, eps and the systems' offsets (None for one system)."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    n, model = case["n"], case["model"]
    if model == "ensemble":
        # system sizes log-uniform in 256..65536 (one set of sizes for every
        # seed), softening 1 / (4 N^(1/3))
        u = np.random.Generator(np.random.PCG64(n)).uniform(math.log(256), math.log(65537), n)
        sizes = np.clip(np.floor(np.exp(u)).astype(np.int64), 256, 65536)
        off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
        per = torch.repeat_interleave(torch.from_numpy(sizes), torch.from_numpy(sizes)).to(DEV).to(F64)
        pos, vel = _plummer(gen, int(off[-1]))
        return pos, vel, 1.0 / per, 0.25 * per ** (-1.0 / 3.0), off
    if model == "cube":
        pos = _uniform(gen, n, 3)
        vel = torch.zeros_like(pos)
    else:
        pos, vel = {"plummer": _plummer, "hernquist": _hernquist, "clumpy": _clumpy}[model](gen, n)
    mass = torch.full((n,), 1.0 / n, dtype=F64, device=DEV)
    return pos.contiguous(), vel.contiguous(), mass, torch.full((n,), case.get("eps") or 1e-3, dtype=F64, device=DEV), None


def _radii(case, pos):
    """Cutoff radii of the short-range mode: 4.2 mean separations of the
    uniform cube, and a radius growing outwards in a cluster."""
    n = pos.shape[0]
    gen = torch.Generator(device=DEV)
    gen.manual_seed(n)
    jitter = 0.9 + 0.2 * _uniform(gen, n)
    if case["model"] == "cube":
        return 4.2 * n ** (-1.0 / 3.0) * jitter
    return 2.6 * n ** (-1.0 / 3.0) * (1.0 + pos.norm(dim=1)) ** 1.5 * jitter


def _rows(case):
    return (np.arange(case["rows"], dtype=np.int64) * case["n"]) // case["rows"]


# --------------------------------------------------------------- the calls

class State:
    """A program's handles and buffers; its destructor closes the handles."""

    def __init__(self, case):
        self.case = case
        self.ctx = self.ps = self.tree = self.law = None

    def __del__(self):
        for h in (self.law, self.tree, self.ps, self.ctx):
            if h is not None:
                h.close()


def prepare(case, seed):
    s = State(case)
    op = case["op"]
    pos, vel, mass, eps, off = _inputs(case, seed)
    if op == "sort":
        s.x, s.y, s.z = (pos[:, k].contiguous() for k in range(3))
        s.keys = torch.empty(case["n"], dtype=torch.int64, device=DEV)
        s.perm = torch.empty(case["n"], dtype=torch.int32, device=DEV)
        return s
    n = pos.shape[0]
    torch.cuda.synchronize()
    s.ctx = G.Context(0)
    s.ps = G.ParticleSystem(s.ctx, n)
    if op == "direct":
        s.rows = _rows(case)
        s.ps.set(pos, vel, mass, eps)
        return s
    s.tree = G.Tree(s.ctx, theta=case.get("theta", 0.5), n_leaf=case["n_leaf"], n_grp=case["n_grp"],
                    quad=case.get("quad", False), fp64=case.get("fp64", False))
    if op == "force":
        host = case["where"] == "host"
        s.data = [t.cpu().pin_memory() if host else t for t in (pos, vel, mass, eps)]
        out = dict(dtype=F64, pin_memory=True) if host else dict(dtype=F64, device=DEV)
        s.acc, s.pot = torch.empty(n, 3, **out), torch.empty(n, **out)
        return s
    if off is not None:
        s.ps.set_systems(off)
    s.ps.set(pos, vel, mass, eps)
    if op == "neighbours":
        s.h = _radii(case, pos)
        torch.cuda.synchronize()
    elif op == "userlaw":
        s.law = G.UserLaw(s.ctx, LAW)
        s.out = torch.zeros(n, 4, dtype=torch.float32, device=DEV)
    else:
        s.tree.calc_force_all_and_write_back(s.ps)  # an integration starts from valid forces
        s.pos, s.vel, s.acc = (torch.empty(n, 3, dtype=F64, device=DEV) for _ in range(3))
        s.pot = torch.empty(n, dtype=F64, device=DEV)
    return s


def run(s):
    case = s.case
    op = case["op"]
    if op == "sort":
        G.fdps_morton_sort_noalloc(s.x, s.y, s.z, case["n"], s.keys, s.perm, torch.cuda.current_stream().cuda_stream)
        return {"keys": s.keys, "perm": s.perm}
    if op == "force":
        s.ps.set(*s.data)
        s.tree.calc_force_all_and_write_back(s.ps)
        G.fdps_psys_get(s.ctx.h, s.ps.h, None, None, s.acc, s.pot)
        return {"acc": s.acc, "pot": s.pot}
    if op == "neighbours":
        fixed = case["mode"] == G.FDPS_CUTOFF_FIXED
        counts, rho, info = s.tree.neighbors(s.ps, case["mode"], None if fixed else s.h, _fixed_radius(case) if fixed else 0.0)
        return {"counts": counts, "rho": rho, "pairs": int(info[0])}
    if op == "userlaw":
        s.tree.build_lists(s.ps)
        s.law.run(s.tree, s.ps, s.out)
        return {"force": s.out}
    if op == "direct":
        acc, pot = s.ps.direct(s.rows)
        return {"acc": acc, "pot": pot}
    if op == "step":
        s.tree.step(s.ps, case["dt"])
    else:
        s.tree.run(s.ps, case["dt"], case["steps"])
    G.fdps_psys_get(s.ctx.h, s.ps.h, s.pos, s.vel, s.acc, s.pot)
    return {"pos": s.pos, "vel": s.vel, "acc": s.acc, "pot": s.pot}


def _fixed_radius(case):
    return (4.2 if case["model"] == "cube" else 4.0) * case["n"] ** (-1.0 / 3.0)


# ------------------------------------------------------------ work, tolerance

def _list_length(n, n_grp, theta):
    """Mean interaction-list length: eq. nlist_long of Sect. 5.5 with half the
    largest group size as the mean one."""
    g = min(0.5 * n_grp, float(n))
    far = max(2.0, theta / 2.8 * (n ** (1 / 3) - g ** (1 / 3)))
    length = g + 14 * g ** (2 / 3) / theta + 21 * math.pi * g ** (1 / 3) / theta ** 2 \
        + 28 * math.pi / (3 * theta ** 3) * math.log2(far)
    return min(float(n), length)


def _interactions(case):
    """Interactions of one force calculation (particles or cells acting on a
    particle)."""
    if case["model"] == "ensemble":
        # mean size of a log-uniform system 256..65536: (65536 - 256) / ln 256
        per = 65280.0 / math.log(256.0)
        return case["n"] * per * _list_length(per, case["n_grp"], case["theta"])
    return case["n"] * _list_length(case["n"], case["n_grp"], case["theta"])


def _particles(case):
    return case["n"] * 65280.0 / math.log(256.0) if case["model"] == "ensemble" else float(case["n"])


def work(case):
    op, n = case["op"], _particles(case)
    if op == "sort":
        return {"bytes": n * (24 + 12), "flops": n * 6}
    if op == "neighbours":
        # 20 operations on each of the neighbours, positions, masses and radii in, counts and densities out
        k = 310.0 if case["model"] == "cube" else 150.0
        return {"bytes": n * (40 + 12), "flops": n * k * 20}
    if op == "direct":
        return {"bytes": n * 40 + case["rows"] * 32, "flops": n * case["rows"] * 20.0}
    # a particle term takes about 20 operations (3 differences, r^2, the
    # root, 3 products, 4 sums), a quadrupole superparticle 50; three
    # quarters of a list are superparticles
    per = 0.25 * 20 + 0.75 * (50 if case["quad"] else 20)
    pairs = _interactions(case)
    if op == "force":
        return {"bytes": n * (64 + 32), "flops": pairs * per}
    if op == "userlaw":
        return {"bytes": n * (40 + 16), "flops": pairs * per}
    steps = case.get("steps", 1)
    return {"bytes": n * (steps * 2 * 80 + 80), "flops": steps * pairs * per}


def tolerance(case):
    """About four times the largest error against `exact` that was seen over
    these ranges (36 cases)."""
    op = case["op"]
    if op == "sort":
        return "exact"
    if op == "neighbours":
        # counts are decided in 64 bits; densities are 32-bit sums
        return {"rel": 1e-6, "max": 1e-5, "differ": 0.0}
    if case.get("fp64"):
        return {"rel": 1e-13, "max": 1e-12}
    if op == "direct":
        return {"rel": 4e-7, "max": 2e-6}
    if op == "userlaw":
        # the law's own plain 32-bit sums over a few thousand entries
        return {"rel": 5e-6, "max": 3e-5}
    if op == "run":
        # close encounters of small clusters amplify the rounding of a step
        return {"rel": 1e-5, "max": 2e-4}
    return {"rel": 5e-6, "max": 1.5e-4}


# ------------------------------------------------------------------- exact

def _tree(pos, mass, sysid, n_sys, n_leaf, n_grp):
    """The octree of the documented reading: per-level nodes over the sorted
    particles, their moments, and the i-groups.  Returns a dict of tensors;
    `order` sorts the particles by (system, key)."""
    n = pos.shape[0]
    lo = torch.stack([_segmin(pos[:, a], sysid, n_sys) for a in range(3)], 1)
    hi = torch.stack([-_segmin(-pos[:, a], sysid, n_sys) for a in range(3)], 1)
    L = (hi - lo).max(1).values
    L = torch.where(L > 0, L, torch.ones_like(L))
    s = 2.0 ** MAX_LEVEL / L
    q = torch.floor((pos - lo[sysid]) * s[sysid][:, None]).clamp(0, 2 ** MAX_LEVEL - 1).to(torch.int64)
    key = torch.zeros(n, dtype=torch.int64, device=pos.device)
    for b in range(MAX_LEVEL):
        for a in range(3):
            key |= ((q[:, a] >> b) & 1) << (3 * b + 2 - a)
    key, order = torch.sort(key, stable=True)
    if n_sys > 1:
        st, o2 = torch.sort(sysid[order], stable=True)
        order, key = order[o2], key[o2]
    else:
        st = sysid
    p, m, q = pos[order], mass[order], q[order]
    idx = torch.arange(n, device=pos.device)
    t = dict(order=order, pos=p, mass=m, q=q, sys=st, L=L)
    node = {k: [] for k in ("level", "first", "count", "leaf", "com", "quad", "qlo", "sys", "child", "nchild")}
    alive = torch.ones(n, dtype=torch.bool, device=pos.device)  # inside a node of this level
    grp = torch.full((n,), -1, dtype=torch.int64, device=pos.device)
    parent_of = None  # node id of the parent of each particle
    base = 0
    for level in range(MAX_LEVEL + 1):
        pre = key >> (3 * (MAX_LEVEL - level))
        brk = torch.ones(n, dtype=torch.bool, device=pos.device)
        brk[1:] = (pre[1:] != pre[:-1]) | (st[1:] != st[:-1])
        brk &= alive
        first = idx[brk]
        if first.numel() == 0:
            break
        rank = torch.cumsum(brk.to(torch.int64), 0) - 1
        rank = torch.where(alive, rank, torch.zeros_like(rank))
        sel = idx[alive]
        k = rank[sel]
        cnt = torch.zeros(first.numel(), dtype=torch.int64, device=pos.device).index_add_(0, k, torch.ones_like(k))
        leaf = (cnt <= n_leaf) | (level == MAX_LEVEL)
        M = torch.zeros(first.numel(), dtype=F64, device=pos.device).index_add_(0, k, m[sel])
        S = torch.zeros(first.numel(), 3, dtype=F64, device=pos.device).index_add_(0, k, m[sel, None] * p[sel])
        com = torch.where(M[:, None] > 0, S / M[:, None], torch.zeros_like(S))
        d = p[sel] - com[k]
        r2 = (d * d).sum(1)
        Q = torch.stack([3 * d[:, a] * d[:, b] - (r2 if a == b else 0.0)
                         for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))], 1) * m[sel, None]
        Q = torch.zeros(first.numel(), 6, dtype=F64, device=pos.device).index_add_(0, k, Q)
        w = MAX_LEVEL - level
        if parent_of is not None:
            par = parent_of[first]
            nchild.index_add_(0, par, torch.ones_like(par))
            child.scatter_reduce_(0, par, base + torch.arange(first.numel(), device=pos.device), "amin")
        for name, v in (("level", torch.full_like(first, level)), ("first", first), ("count", cnt), ("leaf", leaf),
                        ("com", torch.cat([com, M[:, None]], 1)), ("quad", Q), ("qlo", (q[first] >> w) << w), ("sys", st[first])):
            node[name].append(v)
        child = torch.full_like(first, 1 << 60)
        nchild = torch.zeros_like(first)
        node["child"].append(child)
        node["nchild"].append(nchild)
        # groups: maximal cells of at most n_grp particles
        isg = ((cnt <= n_grp) | leaf)[rank] & alive & (grp < 0)
        grp = torch.where(isg, base + rank, grp)
        child = node["child"][-1]
        # particles below internal nodes stay alive; ids local to this level
        parent_of = torch.where(alive, rank, torch.zeros_like(rank))
        alive = alive & ~leaf[rank]
        base += first.numel()
    for name, v in node.items():
        t["n_" + name] = torch.cat(v)
    gfirst = idx[torch.cat([torch.ones(1, dtype=torch.bool, device=pos.device), grp[1:] != grp[:-1]])]
    t["g_first"] = gfirst
    t["g_count"] = torch.diff(torch.cat([gfirst, torch.tensor([n], device=pos.device)]))
    gi = torch.cumsum(torch.zeros(n, dtype=torch.int64, device=pos.device).index_fill_(0, gfirst, 1), 0) - 1
    ng = gfirst.numel()
    t["g_lo"] = torch.stack([_segmin(p[:, a], gi, ng) for a in range(3)], 1)
    t["g_hi"] = torch.stack([-_segmin(-p[:, a], gi, ng) for a in range(3)], 1)
    t["g_qlo"] = torch.stack([_segmin(q[:, a], gi, ng) for a in range(3)], 1)
    t["g_qhi"] = torch.stack([-_segmin(-q[:, a], gi, ng) for a in range(3)], 1)
    t["roots"] = n_sys
    return t


def _segmin(v, idx, n):
    big = torch.full((n,), float("inf") if v.is_floating_point() else 1 << 60, dtype=v.dtype, device=v.device)
    return big.scatter_reduce_(0, idx, v, "amin")


def _expand(first, count):
    """Concatenated ranges first[k] .. first[k] + count[k] - 1 and the k of
    every element."""
    k = torch.repeat_interleave(torch.arange(first.numel(), device=first.device), count)
    start = torch.cumsum(count, 0) - count
    return first[k] + torch.arange(k.numel(), device=first.device) - start[k], k


def _lists(t, theta, g0, g1):
    """Sources of groups g0 .. g1 - 1, sorted by group: indices below n are
    particles, n + node id superparticles.  Returns (source, group - g0)."""
    n = t["pos"].shape[0]
    g = torch.arange(g0, g1, device=t["pos"].device)
    gsys = t["sys"][t["g_first"][g]]
    node = gsys.clone()  # the roots are nodes 0 .. n_sys - 1
    src, own = [], []
    while node.numel():
        w = (1 << (MAX_LEVEL - t["n_level"][node])) - 1
        qlo = t["n_qlo"][node]
        meets = ((qlo <= t["g_qhi"][g]) & (qlo + w[:, None] >= t["g_qlo"][g])).all(1)
        com = t["n_com"][node]
        d2 = torch.zeros(node.numel(), dtype=F64, device=com.device)
        for a in range(3):
            below, above = t["g_lo"][g, a] - com[:, a], com[:, a] - t["g_hi"][g, a]
            da = torch.where(below > 0, below, torch.where(above > 0, above, torch.zeros_like(above)))
            d2 = d2 + da * da
        ell = torch.ldexp(t["L"][t["n_sys"][node]], -t["n_level"][node])
        opened = meets | (ell * ell >= (theta * theta) * d2)
        leaf = t["n_leaf"][node]
        far = ~opened
        src.append(n + node[far])
        own.append(g[far])
        el = opened & leaf
        p, k = _expand(t["n_first"][node[el]], t["n_count"][node[el]])
        src.append(p)
        own.append(g[el][k])
        it = opened & ~leaf
        node_i, g_i = node[it], g[it]
        node, k = _expand(t["n_child"][node_i], t["n_nchild"][node_i])
        g = g_i[k]
    src, own = torch.cat(src), torch.cat(own) - g0
    own, o = torch.sort(own, stable=True)
    return src[o], own


def _tree_force(pos, mass, eps, off, case):
    """(acc, pot) of the tree force in the caller's order."""
    n = pos.shape[0]
    if off is None:
        sysid, n_sys = torch.zeros(n, dtype=torch.int64, device=pos.device), 1
    else:
        sizes = torch.from_numpy(np.diff(off)).to(pos.device)
        n_sys = sizes.numel()
        sysid = torch.repeat_interleave(torch.arange(n_sys, device=pos.device), sizes)
    t = _tree(pos, mass, sysid, n_sys, case["n_leaf"], case["n_grp"])
    zero = torch.zeros(n, 6, dtype=F64, device=pos.device)
    table = torch.cat([torch.cat([t["pos"], t["mass"][:, None], zero], 1),
                       torch.cat([t["n_com"], t["n_quad"] if case["quad"] else torch.zeros_like(t["n_quad"])], 1),
                       torch.zeros(1, 10, dtype=F64, device=pos.device)])
    none = table.shape[0] - 1  # the padding source: no mass
    e2 = (eps * eps)[t["order"]]
    out = torch.zeros(n, 4, dtype=F64, device=pos.device)
    ng = t["g_first"].numel()
    for g0 in range(0, ng, 4096):
        g1 = min(ng, g0 + 4096)
        src, own = _lists(t, case["theta"], g0, g1)
        length = torch.bincount(own, minlength=g1 - g0)
        start = torch.cumsum(length, 0) - length
        by = torch.argsort(length)
        rows, k = _expand(t["g_first"][g0:g1][by], t["g_count"][g0:g1][by])
        row_len, row_start = length[by][k], start[by][k]
        a = 0
        while a < rows.numel():
            # rows a .. b, their lists padded to the longest (the last row's)
            step = max(1, int(1.2e7 / max(1, int(row_len[min(rows.numel() - 1, a + 4096)]))))
            b = min(rows.numel(), a + step)
            width = int(row_len[b - 1])
            col = torch.arange(width, device=pos.device)[None, :]
            at = row_start[a:b, None] + col
            ids = torch.where(col < row_len[a:b, None], src[at.clamp(max=src.numel() - 1)], none)
            out[rows[a:b]] = _pair_sums(t["pos"][rows[a:b]], e2[rows[a:b]], table[ids], case["quad"])
            a = b
    out[:, 3] += t["mass"] / torch.sqrt(e2)
    back = torch.empty_like(out)
    back[t["order"]] = out
    return back[:, :3].contiguous(), back[:, 3].contiguous()


def _pair_sums(x, e2, s, quad):
    """Accelerations and potentials of rows x [r][3] from sources s [r][k][10]."""
    rx, ry, rz = (x[:, a, None] - s[:, :, a] for a in range(3))
    R2 = rx * rx + ry * ry + rz * rz + e2[:, None]
    Ri = 1.0 / torch.sqrt(R2)
    Ri2 = Ri * Ri
    M = s[:, :, 3]
    c = M * Ri * Ri2
    ph = M * Ri
    if not quad:
        return torch.stack([-(c * rx).sum(1), -(c * ry).sum(1), -(c * rz).sum(1), -ph.sum(1)], 1)
    xx, yy, zz, xy, xz, yz = (s[:, :, 4 + a] for a in range(6))
    Qx, Qy, Qz = xx * rx + xy * ry + xz * rz, xy * rx + yy * ry + yz * rz, xz * rx + yz * ry + zz * rz
    rQr = rx * Qx + ry * Qy + rz * Qz
    R5 = Ri2 * Ri2 * Ri
    c = c + 2.5 * rQr * R5 * Ri2
    ph = ph + 0.5 * rQr * R5
    return torch.stack([(Qx * R5 - c * rx).sum(1), (Qy * R5 - c * ry).sum(1), (Qz * R5 - c * rz).sum(1), -ph.sum(1)], 1)


def _exact_sort(pos):
    n = pos.shape[0]
    lo = pos.min(0).values
    L = (pos.max(0).values - lo).max()
    q = torch.floor((pos - lo) * (2.0 ** MAX_LEVEL / L)).clamp(0, 2 ** MAX_LEVEL - 1).to(torch.int64)
    key = torch.zeros(n, dtype=torch.int64, device=pos.device)
    for b in range(MAX_LEVEL):
        for a in range(3):
            key |= ((q[:, a] >> b) & 1) << (3 * b + 2 - a)
    keys, perm = torch.sort(key, stable=True)
    return {"keys": keys, "perm": perm.to(torch.int32)}


def _wendland(r, h):
    q = r / h
    u = (1.0 - q).clamp(min=0.0)
    return 1365.0 / (64.0 * math.pi * h ** 3) * u ** 8 * (1.0 + 8.0 * q + 25.0 * q * q + 32.0 * q ** 3)


def _exact_neighbours(case, pos, mass, h):
    """Neighbour counts and densities by a search over the cells of a grid
    as wide as the largest cutoff that can apply."""
    n, mode = pos.shape[0], case["mode"]
    if mode == G.FDPS_CUTOFF_FIXED:
        h = torch.full_like(mass, _fixed_radius(case))
    if case["model"] != "cube" and n > 30000:
        return None  # radii of very different sizes: no grid fits
    if case["model"] != "cube":
        cnt, rho = _pairs_of(pos, mass, h, mode, torch.arange(n, device=pos.device),
                             torch.zeros(n, dtype=torch.int64, device=pos.device), torch.full((n,), n, device=pos.device))
    else:
        cell = float(h.max())
        dim = max(1, int(1.0 / cell))
        c = (pos * dim).to(torch.int64).clamp(0, dim - 1)
        flat = (c[:, 0] * dim + c[:, 1]) * dim + c[:, 2]
        flat, o = torch.sort(flat)
        count = torch.bincount(flat, minlength=dim ** 3)
        start = torch.cumsum(count, 0) - count
        p, m, hh, cc = pos[o], mass[o], h[o], c[o]
        cnt_s = torch.zeros(n, dtype=torch.int64, device=pos.device)
        rho_s = torch.zeros(n, dtype=F64, device=pos.device)
        rows = torch.arange(n, device=pos.device)
        # a run of cells along z is one range of the sorted particles
        zlo, zhi = (cc[:, 2] - 1).clamp(min=0), (cc[:, 2] + 1).clamp(max=dim - 1)
        for dx in (-1, 0, 1):
            for dy in (-1, 0, 1):
                x, y = cc[:, 0] + dx, cc[:, 1] + dy
                ok = (x >= 0) & (x < dim) & (y >= 0) & (y < dim)
                k = (x.clamp(0, dim - 1) * dim + y.clamp(0, dim - 1)) * dim
                a, e = start[k + zlo], start[k + zhi] + count[k + zhi]
                dc, dr = _pairs_of(p, m, hh, mode, rows, a, torch.where(ok, e - a, torch.zeros_like(a)))
                cnt_s += dc
                rho_s += dr
        cnt, rho = torch.empty_like(cnt_s), torch.empty_like(rho_s)
        cnt[o], rho[o] = cnt_s, rho_s
    return {"counts": cnt.cpu().numpy().astype(np.uint32), "rho": rho.cpu().numpy(), "pairs": int(cnt.sum())}


def _pairs_of(p, m, h, mode, rows, first, count):
    """Counts and densities of rows from candidates first .. first + count."""
    cnt = torch.zeros(rows.numel(), dtype=torch.int64, device=p.device)
    rho = torch.zeros(rows.numel(), dtype=F64, device=p.device)
    step = max(1, int(2e7 / max(1.0, float(count.to(F64).mean()))))
    for a in range(0, rows.numel(), step):
        i, f, c = rows[a:a + step], first[a:a + step], count[a:a + step]
        col = torch.arange(int(c.max()), device=p.device)[None, :]
        ok = col < c[:, None]
        j = torch.where(ok, f[:, None] + col, 0)
        d = [p[j, k] - p[i, k, None] for k in range(3)]
        r2 = (d[0] * d[0] + d[1] * d[1]) + d[2] * d[2]
        hi, hj = h[i, None].expand_as(r2), h[j]
        cut = hi if mode <= 1 else hj if mode == 2 else torch.maximum(hi, hj)
        nb = ok & (r2 < cut * cut)
        r = torch.sqrt(r2)
        w = 0.5 * (_wendland(r, hi) + _wendland(r, hj)) if mode == 3 else _wendland(r, cut)
        cnt[a:a + step] = nb.sum(1)
        rho[a:a + step] = torch.where(nb, m[j] * w, torch.zeros_like(w)).sum(1)
    return cnt, rho


def exact(case, seed):
    op = case["op"]
    pos, vel, mass, eps, off = _inputs(case, seed)
    if op == "sort":
        return _exact_sort(pos)
    if op == "neighbours":
        return _exact_neighbours(case, pos, mass, _radii(case, pos))
    if op == "direct":
        if case["n"] * case["rows"] > EXACT_PAIRS:
            return None
        rows = torch.from_numpy(_rows(case)).to(pos.device)
        acc, pot = torch.zeros(rows.numel(), 3, dtype=F64, device=pos.device), torch.zeros(rows.numel(), dtype=F64, device=pos.device)
        step = max(1, int(4e7 // pos.shape[0]))
        for a in range(0, rows.numel(), step):
            i = rows[a:a + step]
            d = [pos[None, :, k] - pos[i, k, None] for k in range(3)]
            ri = 1.0 / torch.sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2] + (eps[i] * eps[i])[:, None])
            w = mass[None, :] * ri
            w[torch.arange(i.numel(), device=pos.device), i] = 0.0  # not the particle itself
            pot[a:a + step] = -w.sum(1)
            w = w * ri * ri
            acc[a:a + step] = torch.stack([(w * x).sum(1) for x in d], 1)
        return {"acc": acc.cpu().numpy(), "pot": pot.cpu().numpy()}
    forces = {"step": 2, "run": case.get("steps", 1) + 1}.get(op, 1)
    if forces * _interactions(case) > EXACT_PAIRS:
        return None
    acc, pot = _tree_force(pos, mass, eps, off, case)
    if op == "userlaw":  # the law sees each particle's own entry
        return {"force": torch.cat([acc, (pot - mass / eps)[:, None]], 1)}
    if op == "force":
        return {"acc": acc, "pot": pot}
    dt = case["dt"]
    for _ in range(forces - 1):
        vel = vel + 0.5 * dt * acc
        pos = pos + dt * vel
        acc, pot = _tree_force(pos, mass, eps, off, case)
        vel = vel + 0.5 * dt * acc
    return {"pos": pos, "vel": vel, "acc": acc, "pot": pot}
