"""Performance cases of the pairwise-force library: what its users call, over
the range of sizes they call it with.

A case is one call sequence of a simulation or fitting program through the
package's public entry points: all-pairs gravity from a few thousand to a
million bodies, individual time steps (few due particles against a large
set), the periodic cutoff force alone and with the particle mesh, the tree
with both kinds of node moments, caller-made interaction lists, and the
forward and backward pass of a training step.

Positions and masses are FP64, as the library takes them. The library sums
pair terms formed in FP32 (its documented accuracy against FP64 is 2e-6
median, 1e-4 at most), so the programs here keep the acceleration and the
potential in single precision in their particle store, as collisionless
N-body codes do, and run() hands them over there: every pass ends with that
store. The fitting cases train FP32 parameters and return FP32 gradients.
"""

from __future__ import annotations

import math

import numpy as np
import torch

import paper_1203_4037_gb300 as pg

DEV = "cuda"
F64 = torch.float64
RS_OVER_EPS = 16.0        # cutoff shape: eps = r_s / 16
RCUT_OVER_RS = 4.5


def listed():
    return [
        # the accuracy workload's 4096-body Plummer sphere, replayed from a
        # graph: one step of a small direct-sum integration, all latency
        dict(name="direct_4096", kind="newton", n=4096, model="plummer", eps=1 / 64, host=False),
        # a ragged mid-size direct sum by the GRAPE call sequence, host
        # arrays in and out
        dict(name="direct_host_30011", kind="newton", n=30011, model="mix", eps=1e-3, host=True),
        # the headline direct sum: half Plummer sphere, half uniform cube
        dict(name="direct_2e20", kind="newton", n=1 << 20, model="mix", eps=1e-3, host=False),
        # individual time steps: the few particles due now against all others
        dict(name="block_16_on_2e20", kind="block", ni=16, nj=1 << 20, eps=1e-3),
        # a larger block of due particles, ragged
        dict(name="block_1000_on_2e20", kind="block", ni=1000, nj=1 << 20, eps=1e-3),
        # PP alone: the tabulated cutoff force on a clustered periodic box
        dict(name="cells_2e21", kind="cells", n=1 << 21, mesh=256, F=8, pm=False),
        # a full PP + PM force evaluation at a ragged size on a smaller mesh
        dict(name="pppm_250007", kind="cells", n=250007, mesh=128, F=8, pm=True),
        # the tree code's force step, monopole moments
        dict(name="tree_2e20", kind="tree", n=1 << 20, model="plummer", ncrit=256, quad=False, eps=1e-3),
        # the same with quadrupole moments at a ragged size
        dict(name="tree_quad_300007", kind="tree", n=300007, model="mix", ncrit=256, quad=True, eps=1e-3),
        # a host tree code's own interaction lists, kept for several steps
        dict(name="lists_4000", kind="groups", n=1 << 20, ngroups=4000, eps=1e-3),
        # training step through softened gravity (forward and backward)
        dict(name="fit_newton_40009", kind="grad", n=40009, table=False, eps=1 / 64, r_cut=0.1, E=3, F=5),
        # fitting the knots of a cutoff force
        dict(name="fit_table_65536", kind="grad", n=65536, table=True, eps=1 / 64, r_cut=0.1, E=3, F=5),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["newton", "newton", "block", "block", "cells", "pppm", "tree", "groups", "grad", "grad"])
    if kind == "newton":
        n = _logint(rng, 1000, 1 << 19)
        return dict(kind="newton", n=n, model=rng.choice(["plummer", "mix"]),
                    eps=rng.choice([1 / 64, 1e-2, 1e-3]), host=rng.random() < 0.3)
    if kind == "block":
        return dict(kind="block", ni=_logint(rng, 1, 4000), nj=_logint(rng, 1 << 18, 1 << 20),
                    eps=rng.choice([1 / 64, 1e-3]))
    if kind in ("cells", "pppm"):
        mesh = rng.choice([64, 128, 256])
        return dict(kind="cells", n=int(mesh ** 3 // 8 * rng.uniform(0.25, 0.99)), mesh=mesh,
                    F=rng.choice([6, 7, 8]), pm=kind == "pppm")
    if kind == "tree":
        return dict(kind="tree", n=_logint(rng, 1 << 15, (1 << 20) - 1), model=rng.choice(["plummer", "mix"]),
                    ncrit=rng.choice([64, 128, 256]), quad=rng.random() < 0.5, eps=rng.choice([1e-2, 1e-3]))
    if kind == "groups":
        return dict(kind="groups", n=_logint(rng, 1 << 18, 1 << 20), ngroups=_logint(rng, 500, 4000),
                    eps=rng.choice([1e-2, 1e-3]))
    return dict(kind="grad", n=_logint(rng, 3000, 65535), table=rng.random() < 0.5, eps=rng.choice([1 / 64, 1e-2]),
                r_cut=rng.choice([0.1, 0.2]), E=3, F=rng.choice([5, 6]))


# ------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=F64)


def _isotropic(g, n):
    mu = 2 * _rand(g, n) - 1
    ph = 2 * math.pi * _rand(g, n)
    st = torch.sqrt(torch.clamp(1 - mu * mu, min=0))
    return torch.stack([st * torch.cos(ph), st * torch.sin(ph), mu], 1)


def _plummer(g, n):
    """Plummer sphere of scale 1 out to 99.9 % of its mass."""
    X = 0.999 * (1 - _rand(g, n))
    r = 1 / torch.sqrt(X ** (-2 / 3) - 1)
    return (r[:, None] * _isotropic(g, n)).contiguous()


def _particles(g, n, model):
    """(x, m): an equal-mass Plummer sphere, or a shuffled mix of half a
    Plummer sphere and half a uniform cube of side 4 with log-uniform masses."""
    if model == "plummer":
        return _plummer(g, n), torch.full((n,), 1.0 / n, device=DEV, dtype=F64)
    nh = n // 2
    x = torch.cat([_plummer(g, nh), 4 * _rand(g, n - nh, 3) - 2])
    m = torch.exp(math.log(1e-7) + math.log(100.0) * _rand(g, n))
    p = torch.randperm(n, generator=g, device=DEV)
    return x[p].contiguous(), (m / m.sum())[p].contiguous()


def _clustered(g, n, periodic):
    """Unit box: 70 % uniform, 30 % in 200 Gaussian clumps of width 0.005."""
    nc = int(round(0.3 * n))
    centres = _rand(g, 200, 3)
    off = torch.randn(nc, 3, generator=g, device=DEV, dtype=F64)
    xc = centres[torch.arange(nc, device=DEV) % 200] + 0.005 * off
    if periodic:
        xc = xc - torch.floor(xc)
        xc = torch.where(xc >= 1.0, torch.zeros_like(xc), xc)
    x = torch.cat([_rand(g, n - nc, 3), xc])
    p = torch.randperm(n, generator=g, device=DEV)
    return x[p].contiguous(), torch.full((n,), 1.0 / n, device=DEV, dtype=F64)


def _morton(x):
    lo = x.min(0).values
    span = float((x.max(0).values - lo).max()) or 1.0
    q = ((x - lo) / span * ((1 << 20) - 1)).to(torch.int64)
    key = torch.zeros(x.shape[0], dtype=torch.int64, device=x.device)
    for b in range(20):
        for a in range(3):
            key |= ((q[:, a] >> b) & 1) << (3 * b + 2 - a)
    return torch.argsort(key, stable=True)


def _lists(g, n, ngroups):
    """Tree-style groups of 16 to 512 i-particles, each with a list of 1024 to
    16384 j: 70 % a Morton window around the group, 30 % monopoles of runs of
    particles spread over the set. The lists' sizes belong to the case, the
    particles to the seed."""
    x, m = _clustered(g, n, False)
    o = _morton(x)
    x, m = x[o].contiguous(), m[o].contiguous()
    nm = n // 4
    run = torch.randint(8, 65, (nm,), generator=g, device=DEV)
    start = torch.sort(torch.randint(0, n - 64, (nm,), generator=g, device=DEV)).values
    cm = torch.cat([torch.zeros(1, device=DEV, dtype=F64), torch.cumsum(m, 0)])
    cx = torch.cat([torch.zeros(1, 3, device=DEV, dtype=F64), torch.cumsum(m[:, None] * x, 0)])
    mm = cm[start + run] - cm[start]
    xm = (cx[start + run] - cx[start]) / mm[:, None]
    r = np.random.Generator(np.random.PCG64(n + ngroups))

    def logint(lo, hi):
        return np.clip(np.exp(r.uniform(np.log(lo), np.log(hi + 1), ngroups)).astype(np.int64), lo, hi)

    ni, nj = logint(16, 512), logint(1024, 16384)
    gs = (np.arange(ngroups, dtype=np.int64) * (n - 512)) // ngroups
    i_off = np.concatenate([[0], np.cumsum(ni)])
    j_off = np.concatenate([[0], np.cumsum(nj)])
    i_src = np.repeat(gs - i_off[:-1], ni) + np.arange(i_off[-1])
    npart = np.rint(0.7 * nj).astype(np.int64)
    w0 = np.clip(gs + ni // 2 - npart // 2, 0, n - npart)
    phase = r.integers(0, nm, ngroups)
    pos = np.arange(j_off[-1]) - np.repeat(j_off[:-1], nj)
    nmono = np.repeat(np.maximum(nj - npart, 1), nj)
    mono = n + (np.repeat(phase, nj) + (pos - np.repeat(npart, nj)) * nm // nmono) % nm
    jlist = np.where(pos < np.repeat(npart, nj), np.repeat(w0, nj) + pos, mono).astype(np.int32)
    return dict(xi=x[torch.from_numpy(i_src).to(DEV)].contiguous(), xj=torch.cat([x, xm]).contiguous(),
                mj=torch.cat([m, mm]).contiguous(), i_off=i_off, j_off=j_off, jlist=jlist)


def _knots(E, F):
    """The table's knots in s: the FP32 patterns from 2.0 in steps of 2^(23-F)."""
    k = np.arange(1 << (E + F), dtype=np.uint32)
    return (np.uint32(0x40000000) + (k << np.uint32(23 - F))).view(np.float32).astype(np.float64)


def _split_values(E, F, r_cut, rs, eps):
    """Knot values (FP32) of the Gaussian split's short-range shape."""
    s = torch.from_numpy(_knots(E, F))
    r = r_cut * torch.sqrt((s - 2) / (s[-1] - 2))
    g = (torch.special.erfc(r / (2 * rs)) + r / (rs * math.sqrt(math.pi)) * torch.exp(-r * r / (4 * rs * rs)))
    return (g * (r * r + eps * eps) ** -1.5).to(torch.float32).numpy()


def _inputs(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    if kind in ("newton", "tree"):
        x, m = _particles(g, case["n"], case["model"])
        return dict(x=x, m=m)
    if kind == "block":
        xj, mj = _particles(g, case["nj"], "mix")
        # the due particles are the ones deepest in the sphere's core, at
        # positions between those of the set
        xi = _plummer(g, 20 * case["ni"] + 100)
        xi = xi[torch.argsort((xi * xi).sum(1))[:case["ni"]]].contiguous()
        return dict(xi=xi, xj=xj, mj=mj)
    if kind == "cells":
        x, m = _clustered(g, case["n"], True)
        rs = 1.0 / case["mesh"]
        return dict(x=x, m=m, rs=rs, r_cut=RCUT_OVER_RS * rs,
                    v=_split_values(4, case["F"], RCUT_OVER_RS * rs, rs, rs / RS_OVER_EPS))
    if kind == "groups":
        return _lists(g, case["n"], case["ngroups"])
    # training: FP32 parameters, FP64 inside the force call, a given
    # gradient of the loss with respect to the accelerations
    x = _plummer(g, case["n"]).to(torch.float32)
    m = torch.full((case["n"],), 1.0 / case["n"], device=DEV) * (0.5 + torch.rand(case["n"], generator=g, device=DEV))
    d = dict(x=x, m=m, w=_isotropic(g, case["n"]))
    if case["table"]:
        v = _split_values(case["E"], case["F"], case["r_cut"], case["r_cut"] / RCUT_OVER_RS, case["eps"])
        d["v"] = torch.from_numpy(v).to(DEV)
    return d


# ------------------------------------------------------------------ the cases

def _store(n):
    """The library's FP64 output (a, phi in one buffer) and the program's FP32 particle store."""
    out = torch.empty(4 * n, device=DEV, dtype=F64)
    return dict(out=out, a=out[:3 * n].view(n, 3), phi=out[3 * n:], acc=torch.empty(4 * n, device=DEV))


def prepare(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    s = dict(case=case, **d)
    if kind == "grad":
        for k in ("x", "m", "v"):
            if k in s:
                s[k] = s[k].requires_grad_(True)
        return s
    c = s["ctx"] = pg.Context(0)
    c.set_stream(torch.cuda.current_stream().cuda_stream)
    if kind == "newton":
        c.set_eps(case["eps"])
        c.set_self(True)
        if case["host"]:
            s["x"], s["m"] = d["x"].cpu().numpy(), d["m"].cpu().numpy()
        else:
            c.set_graph(True)
            s.update(_store(case["n"]))
    elif kind == "block":
        c.set_eps(case["eps"])
        c.set_j_dev(d["xj"], d["mj"])
        c.set_graph(True)
        s.update(_store(case["ni"]))
    elif kind == "cells":
        c.set_mode(pg.PG_TABLE)
        c.set_table_values(d["v"], d["r_cut"], 4, case["F"])
        c.set_self(True)
        c.set_periodic(1.0)
        if case["pm"]:
            c.set_pm(case["mesh"], pg.PG_SPLIT_GAUSS, d["rs"])
        c.set_graph(True)
        s.update(_store(case["n"]))
    elif kind == "tree":
        c.set_eps(case["eps"])
        c.set_self(True)
        c.set_tree(0.75, case["ncrit"], 8, quadrupole=case["quad"])
        s.update(_store(case["n"]))
    else:
        c.set_eps(case["eps"])
        c.set_j_dev(d["xj"], d["mj"])
        c.set_i_dev(d["xi"])
        c.set_groups(d["i_off"], d["j_off"], d["jlist"])
        c.set_graph(True)
        s.update(_store(d["xi"].shape[0]))
    return s


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "grad":
        from paper_1203_4037_gb300.autograd import newton_force, table_force
        x, m = s["x"].to(F64), s["m"].to(F64)
        if case["table"]:
            a = table_force(x, m, s["v"], case["r_cut"], case["E"], case["F"])
            grads = torch.autograd.grad(a, (s["x"], s["m"], s["v"]), s["w"])
        else:
            a = newton_force(x, m, case["eps"])
            grads = torch.autograd.grad(a, (s["x"], s["m"]), s["w"])
        return [a.detach().to(torch.float32), *grads]
    c = s["ctx"]
    if kind == "newton" and case["host"]:
        a, phi = c.forces(s["x"], s["x"], s["m"])
        return [a.astype(np.float32), phi.astype(np.float32)]
    if kind == "block":
        c.set_i_dev(s["xi"])
    elif kind == "groups":
        c.set_j_dev(s["xj"], s["mj"])
        c.set_i_dev(s["xi"])
    else:
        c.set_j_dev(s["x"], s["m"])
        c.set_i_dev(s["x"])
    phi = None if kind == "cells" and not case["pm"] else s["phi"]
    c.run_dev(s["a"], phi)
    if phi is None:          # the cutoff force alone has no potential
        n3 = s["a"].numel()
        return [s["acc"][:n3].copy_(s["out"][:n3]).view(-1, 3)]
    s["acc"].copy_(s["out"])
    n = s["a"].shape[0]
    return [s["acc"][:3 * n].view(n, 3), s["acc"][3 * n:]]


# ------------------------------------------------------------------ work

def _clump_pairs(n, r_cut):
    """Expected ordered pairs closer than r_cut in the clustered box."""
    M = 0.3 * n / 200
    t = r_cut / (0.005 * math.sqrt(2.0))
    inside = math.erf(t / math.sqrt(2)) - math.sqrt(2 / math.pi) * t * math.exp(-t * t / 2)
    vol = 4 / 3 * math.pi * r_cut ** 3
    return 200 * M * M * inside + n * n * (0.49 + 0.42 + 0.09) * vol


def work(case):
    """Particles in, forces out, and the pair terms: 20 operations for a
    softened Newton pair with its potential (three differences, r^2, inverse
    square root, m/r, m/r^3, four sums), 17 for a tabulated pair."""
    kind = case["kind"]
    if kind == "newton":
        return dict(bytes=64.0 * case["n"], flops=20.0 * case["n"] ** 2)
    if kind == "block":
        return dict(bytes=32.0 * case["nj"] + 56.0 * case["ni"], flops=20.0 * case["ni"] * case["nj"])
    if kind == "cells":
        n, N3 = case["n"], float(case["mesh"] ** 3)
        pairs = 17.0 * _clump_pairs(n, RCUT_OVER_RS / case["mesh"])
        if not case["pm"]:
            return dict(bytes=56.0 * n, flops=pairs)
        # the mesh once through the transforms (one forward, four inverse),
        # 27-point assignment and interpolation of four fields
        return dict(bytes=64.0 * n + 20.0 * N3, flops=pairs + 12.5 * N3 * math.log2(N3) + 27.0 * 10 * n)
    if kind == "tree":
        # about 110 list entries per octave of n at theta = 0.75 and groups of
        # a few hundred (quadrupoles: three pseudo-particles per node)
        return dict(bytes=64.0 * case["n"],
                    flops=20.0 * case["n"] * 90.0 * math.log2(case["n"]) * (2.0 if case["quad"] else 1.0))
    if kind == "groups":
        ng = case["ngroups"]
        mi, mj = 496 / math.log(32.0), 15360 / math.log(16.0)      # means of the log-uniform sizes
        return dict(bytes=56.0 * ng * mi + 40.0 * case["n"] + 4.0 * ng * mj, flops=20.0 * ng * mi * mj)
    n = case["n"]
    if not case["table"]:
        return dict(bytes=84.0 * n, flops=(20.0 + 36.0) * n * n)
    # every pair is tested in both passes (8 operations); the pairs inside
    # the cutoff also take the table and the sums
    return dict(bytes=84.0 * n + 8.0 * (1 << (case["E"] + case["F"])), flops=2 * 8.0 * n * n)


# ------------------------------------------------------------------ 64 bits

PAIRS = 1 << 26           # pairs of one chunk


def _direct(xi, xj, mj, eps, self_):
    a, p = torch.empty_like(xi), torch.empty_like(xi[:, 0])
    step = max(1, PAIRS // xj.shape[0])
    for b in range(0, xi.shape[0], step):
        d = [xj[None, :, k] - xi[b:b + step, None, k] for k in range(3)]
        ri = torch.rsqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2] + eps * eps)
        if self_:
            r = torch.arange(ri.shape[0], device=DEV)
            ri[r, b + r] = 0
        q = mj[None] * ri
        p[b:b + step] = -q.sum(1)
        q *= ri * ri
        for k in range(3):
            a[b:b + step, k] = (q * d[k]).sum(1)
    return a, p


def _segments(val, counts):
    """Sums of consecutive segments of val, (k, pairs), with the given lengths: (segments, k)."""
    cs = torch.cat([torch.zeros(val.shape[0], 1, device=DEV, dtype=F64), torch.cumsum(val, 1)], 1)
    e = torch.cumsum(counts, 0)
    return (cs[:, e] - cs[:, e - counts]).T


def _chunks(cost):
    """Ranges of consecutive elements of about PAIRS / 2 total cost each."""
    cs = np.cumsum(cost.cpu().numpy())
    b = 0
    while b < len(cs):
        base = cs[b - 1] if b else 0
        e = max(b + 1, int(np.searchsorted(cs, base + PAIRS // 2, side="right")))
        yield b, e
        b = e


def _by_lists(xi, gi, j_off, jlist, xj, mj, eps, own=None):
    """Direct sums over lists: particle k uses list gi[k]; own[k]: the j index left out."""
    n = xi.shape[0]
    a, p = torch.zeros(n, 3, device=DEV, dtype=F64), torch.zeros(n, device=DEV, dtype=F64)
    ln = (j_off[1:] - j_off[:-1])[gi]
    for b, e in _chunks(ln):
        c = ln[b:e]
        k = torch.repeat_interleave(torch.arange(b, e, device=DEV), c)
        pos = torch.arange(k.numel(), device=DEV) - (torch.cumsum(c, 0) - c)[k - b]
        j = jlist[j_off[gi[k]] + pos].to(torch.int64)
        d = xj[j] - xi[k]
        ri = torch.rsqrt((d * d).sum(1) + eps * eps)
        if own is not None:
            ri = torch.where(j == own[k], torch.zeros_like(ri), ri)
        q = mj[j] * ri
        s = _segments(torch.cat([(q * ri * ri) * d.T, q[None]]), c)
        a[b:e], p[b:e] = s[:, :3], -s[:, 3]
    return a, p


def _table_terms(E, F, v, r_cut):
    """s of r^2, and (g, dg/ds, bin, fraction) of s < s_max, from FP32 knot values."""
    s = torch.from_numpy(_knots(E, F)).to(DEV)
    v = torch.as_tensor(v).to(DEV).to(F64)
    slope = (v[1:] - v[:-1]) / (s[1:] - s[:-1])
    kappa = float(s[-1] - 2) / r_cut ** 2

    def at(sv):
        k = torch.clamp(torch.searchsorted(s, sv, right=True) - 1, 0, s.numel() - 2)
        return v[k] + (sv - s[k]) * slope[k], slope[k], k, (sv - s[k]) / (s[k + 1] - s[k])

    return kappa, float(s[-1]), at


def _cells(x, m, r_cut, E, F, v):
    """The periodic (box 1) tabulated force by neighbour cells of side >= r_cut."""
    n, nc = x.shape[0], int(1.0 / r_cut)
    kappa, smax, at = _table_terms(E, F, v, r_cut)
    q = torch.clamp((x * nc).to(torch.int64), 0, nc - 1)
    cell = (q[:, 0] * nc + q[:, 1]) * nc + q[:, 2]
    o = torch.argsort(cell, stable=True)
    xs, ms, qs = x[o], m[o], q[o]
    cnt = torch.bincount(cell, minlength=nc ** 3)
    first = torch.cumsum(cnt, 0) - cnt
    acc = torch.zeros(n, 3, device=DEV, dtype=F64)
    for sx in (-1, 0, 1):
        for sy in (-1, 0, 1):
            for sz in (-1, 0, 1):
                nb = (qs + torch.tensor([sx, sy, sz], device=DEV)) % nc
                nb = (nb[:, 0] * nc + nb[:, 1]) * nc + nb[:, 2]
                c_all = cnt[nb]
                for b, e in _chunks(c_all):
                    c = c_all[b:e]
                    k = torch.repeat_interleave(torch.arange(b, e, device=DEV), c)
                    j = first[nb[k]] + torch.arange(k.numel(), device=DEV) - (torch.cumsum(c, 0) - c)[k - b]
                    d = xs[j] - xs[k]
                    d -= torch.round(d)
                    s = 2 + kappa * (d * d).sum(1)
                    g = torch.where(s < smax, at(s)[0], torch.zeros_like(s)) * ms[j]
                    acc[b:e] += _segments(g * d.T, c)
    out = torch.empty_like(acc)
    out[o] = acc
    return out


def _mesh(x, m, N, rs):
    """TSC mesh forces of the Gaussian split's long range in the unit box."""
    u = x * N
    j0 = torch.floor(u + 0.5)
    d = u - j0
    w = torch.stack([0.5 * (0.5 - d) ** 2, 0.75 - d * d, 0.5 * (0.5 + d) ** 2], 0)     # (3, n, axis)
    idx = [(j0.to(torch.int64) + t) % N for t in (-1, 0, 1)]
    rho = torch.zeros(N ** 3, device=DEV, dtype=F64)
    stencil = [(ix, iy, iz) for ix in range(3) for iy in range(3) for iz in range(3)]

    def at(t):
        ix, iy, iz = t
        cell = (idx[ix][:, 0] * N + idx[iy][:, 1]) * N + idx[iz][:, 2]
        return cell, w[ix][:, 0] * w[iy][:, 1] * w[iz][:, 2]

    for t in stencil:
        cell, wt = at(t)
        rho.index_add_(0, cell, m * wt * float(N) ** 3)
    fk = torch.fft.fftfreq(N, 1.0 / N, device=DEV, dtype=F64)
    win = torch.sinc(fk / N) ** 3
    kx, ky, kz = torch.meshgrid(fk, fk, fk[:N // 2 + 1].abs(), indexing="ij")
    k2 = (2 * math.pi) ** 2 * (kx * kx + ky * ky + kz * kz)
    wx, wy, wz = torch.meshgrid(win, win, win[:N // 2 + 1], indexing="ij")
    G = -4 * math.pi * torch.exp(-k2 * rs * rs) / torch.where(k2 > 0, k2, torch.ones_like(k2)) / (wx * wy * wz) ** 2
    nyq = (kx.abs() == N // 2) | (ky.abs() == N // 2) | (kz == N // 2)
    G = torch.where((k2 == 0) | nyq, torch.zeros_like(G), G)
    phik = torch.fft.rfftn(rho.view(N, N, N)) * G
    fields = [torch.fft.irfftn(-2j * math.pi * k * phik, s=(N, N, N)).reshape(-1) for k in (kx, ky, kz)]
    fields.append(torch.fft.irfftn(phik, s=(N, N, N)).reshape(-1))
    out = torch.zeros(x.shape[0], 4, device=DEV, dtype=F64)
    for t in stencil:
        cell, wt = at(t)
        for k in range(4):
            out[:, k] += wt * fields[k][cell]
    return out[:, :3], out[:, 3]


def _quadrupole_points(com, M, T):
    """Three particles of mass M/3 with the node's mass, centre and trace-free second moment."""
    l, V = (t.to(DEV) for t in torch.linalg.eigh(T.cpu()))
    e1, e2 = V[:, :, 2], V[:, :, 1]
    big = torch.argmax(e1.abs(), 1, keepdim=True)
    e1 = e1 * torch.sign(torch.gather(e1, 1, big))
    a = torch.sqrt(torch.clamp(2 * (l[:, 2] - l[:, 0]) / M, min=0))[:, None] * e1
    b = torch.sqrt(torch.clamp(2 * (l[:, 1] - l[:, 0]) / M, min=0))[:, None] * e2
    h = math.sqrt(3) / 2 * b
    return torch.stack([com + a, com - a / 2 + h, com - a / 2 - h], 1)


def _tree(x, m, eps, theta, ncrit, nleaf, quad):
    """Barnes-Hut forces: octree on 10-bit keys, groups of at most ncrit,
    opening by the distance from a node's centre of mass to the group's box."""
    n = x.shape[0]
    lo = x.min(0).values
    span = float((x.max(0).values - lo).max()) or 1.0
    q = torch.clamp(torch.floor((x - lo) / span * 1024), 0, 1023).to(torch.int64)
    key = torch.zeros(n, dtype=torch.int64, device=DEV)
    for b in range(10):
        for k in range(3):
            key |= ((q[:, k] >> b) & 1) << (3 * b + 2 - k)
    o = torch.argsort(key, stable=True)
    xs, ms, key = x[o], m[o], key[o]
    lev, base = [], 0
    for L in range(11):
        _, inv, cnt = torch.unique_consecutive(key >> (3 * (10 - L)), return_inverse=True, return_counts=True)
        first = torch.cumsum(cnt, 0) - cnt
        M = torch.zeros(cnt.numel(), device=DEV, dtype=F64).index_add_(0, inv, ms)
        com = torch.zeros(cnt.numel(), 3, device=DEV, dtype=F64).index_add_(0, inv, ms[:, None] * xs) / M[:, None]
        lev.append(dict(inv=inv, cnt=cnt, first=first, M=M, com=com, base=base))
        base += cnt.numel()
    g0, gn = [], []
    for L, v in enumerate(lev):
        if L == 0:
            pick = v["cnt"] <= ncrit
        else:
            big = lev[L - 1]["cnt"][lev[L - 1]["inv"][v["first"]]] > ncrit
            pick = big if L == 10 else big & (v["cnt"] <= ncrit)
        g0.append(v["first"][pick])
        gn.append(v["cnt"][pick])
    g0, gn = torch.cat(g0), torch.cat(gn)
    o2 = torch.argsort(g0)
    g0, gn = g0[o2], gn[o2]
    ng = g0.numel()
    gi = torch.repeat_interleave(torch.arange(ng, device=DEV), gn)
    ix = gi[:, None].expand(-1, 3)
    bmin = torch.full((ng, 3), math.inf, device=DEV, dtype=F64).scatter_reduce_(0, ix, xs, "amin")
    bmax = torch.full((ng, 3), -math.inf, device=DEV, dtype=F64).scatter_reduce_(0, ix, xs, "amax")
    eg, ej = [], []
    fg = torch.arange(ng, device=DEV)
    fk = torch.zeros(ng, dtype=torch.int64, device=DEV)
    npseudo = 3 if quad else 1
    for L, v in enumerate(lev):
        first, cnt, com = v["first"][fk], v["cnt"][fk], v["com"][fk]
        apart = (first + cnt <= g0[fg]) | (first >= g0[fg] + gn[fg])
        d = torch.clamp(torch.maximum(bmin[fg] - com, com - bmax[fg]), min=0)
        side = span / (1 << L)
        acc = apart & (side * side < theta * theta * (d * d).sum(1))
        for t in range(npseudo):
            eg.append(fg[acc])
            ej.append(n + (v["base"] + fk[acc]) * npseudo + t)
        leaf = ~acc & ((cnt <= nleaf) | (L == 10))
        c = cnt[leaf]
        eg.append(torch.repeat_interleave(fg[leaf], c))
        ej.append(torch.repeat_interleave(first[leaf] - (torch.cumsum(c, 0) - c), c) +
                  torch.arange(int(c.sum()), device=DEV))
        if L == 10:
            break
        op = ~acc & ~leaf
        f, w = first[op], lev[L + 1]
        c0 = w["inv"][f]
        c = w["inv"][f + cnt[op] - 1] - c0 + 1
        fg = torch.repeat_interleave(fg[op], c)
        fk = torch.repeat_interleave(c0 - (torch.cumsum(c, 0) - c), c) + torch.arange(int(c.sum()), device=DEV)
    eg, ej = torch.cat(eg), torch.cat(ej)
    so = torch.argsort(eg, stable=True)
    ej = ej[so]
    j_off = torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV),
                       torch.cumsum(torch.bincount(eg, minlength=ng), 0)])
    px, pm = [], []
    for v in lev:
        if not quad:
            px.append(v["com"])
            pm.append(v["M"])
            continue
        r = xs - v["com"][v["inv"]]
        T = torch.zeros(v["M"].numel(), 9, device=DEV, dtype=F64)
        T.index_add_(0, v["inv"], ms[:, None] * (r[:, :, None] * r[:, None, :]).reshape(-1, 9))
        one = (v["cnt"] == 1)[:, None]
        T = torch.where(one, torch.zeros_like(T), T).view(-1, 3, 3)
        px.append(_quadrupole_points(v["com"], v["M"], T).reshape(-1, 3))
        pm.append(torch.repeat_interleave(v["M"] / 3, 3))
    a, p = _by_lists(xs, gi, j_off, ej, torch.cat([xs, *px]), torch.cat([ms, *pm]), eps,
                     own=torch.arange(n, device=DEV))
    ao, po = torch.empty_like(a), torch.empty_like(p)
    ao[o], po[o] = a, p
    return ao, po


def _gradients(case, d):
    x, m, w = d["x"].to(F64), d["m"].to(F64), d["w"]
    n = x.shape[0]
    a, dx = torch.empty_like(x), torch.zeros_like(x)
    dm = torch.zeros_like(m)
    if case["table"]:
        nk = 1 << (case["E"] + case["F"])
        kappa, smax, at = _table_terms(case["E"], case["F"], d["v"], case["r_cut"])
        dv = torch.zeros(nk, device=DEV, dtype=F64)
    step = max(1, PAIRS // n)
    for b in range(0, n, step):
        e = min(n, b + step)
        dd = [x[None, :, k] - x[b:e, None, k] for k in range(3)]
        r2 = dd[0] * dd[0] + dd[1] * dd[1] + dd[2] * dd[2]
        i, j = None, None
        if case["table"]:
            r2[torch.arange(e - b, device=DEV), torch.arange(b, e, device=DEV)] = math.inf
            s = 2 + kappa * r2
            i, j = torch.nonzero(s < smax, as_tuple=True)
            s, D = s[i, j], x[j] - x[b + i]
            g, gs, k, t = at(s)
            u = (w[b + i] * D).sum(1)
            a[b:e] = torch.zeros(e - b, 3, device=DEV, dtype=F64).index_add_(0, i, (m[j] * g)[:, None] * D)
            dm.index_add_(0, j, g * u)
            dv += torch.bincount(k, weights=m[j] * u * (1 - t), minlength=nk)
            dv += torch.bincount(k + 1, weights=m[j] * u * t, minlength=nk)
            f = m[j][:, None] * (g[:, None] * w[b + i] + (2 * kappa * gs * u)[:, None] * D)
            dx.index_add_(0, j, f)
            dx.index_add_(0, b + i, -f)
            continue
        ri = torch.rsqrt(r2 + case["eps"] ** 2)
        r = torch.arange(e - b, device=DEV)
        ri[r, b + r] = 0
        ri3 = ri * ri * ri
        u = sum(dd[k] * w[b:e, None, k] for k in range(3))
        dm += (ri3 * u).sum(0)
        q = -3 * u * ri3 * ri * ri * m[None]
        ri3 *= m[None]
        for k in range(3):
            a[b:e, k] = (ri3 * dd[k]).sum(1)
            f = ri3 * w[b:e, None, k] + q * dd[k]
            dx[:, k] += f.sum(0)
            dx[b:e, k] -= f.sum(1)
    return [a, dx, dm, dv] if case["table"] else [a, dx, dm]


def exact(case, seed):
    kind = case["kind"]
    if kind == "newton" and case["n"] > 300000:
        return None
    with torch.no_grad():
        d = _inputs(case, seed)
        if kind == "newton":
            return list(_direct(d["x"], d["x"], d["m"], case["eps"], True))
        if kind == "block":
            return list(_direct(d["xi"], d["xj"], d["mj"], case["eps"], False))
        if kind == "cells":
            a = _cells(d["x"], d["m"], d["r_cut"], 4, case["F"], d["v"])
            if not case["pm"]:
                return [a]
            am, pm = _mesh(d["x"], d["m"], case["mesh"], d["rs"])
            return [a + am, pm]
        if kind == "tree":
            return list(_tree(d["x"], d["m"], case["eps"], 0.75, case["ncrit"], 8, case["quad"]))
        if kind == "groups":
            gi = torch.from_numpy(np.repeat(np.arange(case["ngroups"]), np.diff(d["i_off"]))).to(DEV)
            return list(_by_lists(d["xi"], gi, torch.from_numpy(d["j_off"]).to(DEV),
                                  torch.from_numpy(d["jlist"]).to(DEV), d["xj"], d["mj"], case["eps"]))
        return _gradients(case, d)
