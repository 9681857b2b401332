"""Performance cases of the SFMM gravity solver.

Each case is one pass that a program using this package makes again and again:
a time step's gravity (build + gravity on device arrays), the same step as one
captured graph, a whole ensemble of systems, a solve of host arrays, a few
leapfrog steps.  ``listed()`` and ``draw()`` give the cases, ``prepare()`` what
the program has in hand, ``run()`` one pass, ``work()`` the bytes and
operations it cannot do without, ``exact()`` the same results in float64 from
plain torch, written here from the method (tree, moments, dual-tree walk,
expansions, softened pairs) without the package.

Particle sets follow the test problems: homogeneous and Plummer spheres, two
n = 1.5 polytropes, a clustered cloud, an ensemble of small systems; equal
particle masses and h = 1.2 (m / rho)^(1/3) from the analytic density, so that
neighbouring particles lie inside one another's softening kernels.
"""
import math

import numpy as np
import torch

from paper_2602_05804_gb300 import sfmm

HFACT = 1.2


def _dev():
    return torch.device("cuda:0" if torch.cuda.is_available() else "cpu")


# --------------------------------------------------------------------------
# Cases
# --------------------------------------------------------------------------
def _case(entry, form, profile, n, leaf, theta, order, **more):
    return dict(entry=entry, form=form, profile=profile, n=n, leaf=leaf, theta=theta, order=order, **more)


def listed():
    return [
        # a star cluster or clump handled on its own: latency and launches
        dict(_case("step", "fp32", "uniform", 1000, 16, 0.5, 2), name="step_fp32_uniform_1e3"),
        # the small accuracy configuration: FP64 form on a homogeneous sphere
        dict(_case("step", "fp64", "uniform", 10000, 10, 0.5, 2), name="step_fp64_uniform_1e4"),
        # a mid-size halo at high order and a wide opening angle
        dict(_case("step", "fp32", "plummer", 100003, 16, 0.7, 4), name="step_fp32_plummer_1e5_p4"),
        # the FP64 form at the leaf size that suits it, third order
        dict(_case("step", "fp64", "plummer", 99991, 8, 0.5, 3), name="step_fp64_plummer_1e5_p3"),
        # the benchmark's step: one captured graph per time step
        dict(_case("graph", "fp32", "plummer", 1000000, 16, 0.5, 2), name="graph_fp32_plummer_1e6"),
        # the accurate end of the opening angles, ordinary calls
        dict(_case("step", "fp32", "plummer", 1000000, 16, 0.3, 2), name="step_fp32_plummer_1e6_t03"),
        # the benchmark's step in the FP64 form
        dict(_case("step", "fp64", "plummer", 1000000, 16, 0.5, 2), name="step_fp64_plummer_1e6"),
        # two stars, wide range of h at their surfaces
        dict(_case("step", "fp32", "binary", 2000000, 16, 0.5, 2), name="step_fp32_binary_2e6"),
        # 256 independent systems of 10^3 .. 10^5 particles in one launch
        dict(_case("graph", "fp32", "ensemble", 256, 0, 0.5, 2), name="graph_fp32_ensemble_256"),
        # the largest set: a halo with dense clumps
        dict(_case("step", "fp32", "cloud", 16000000, 16, 0.5, 2), name="step_fp32_cloud_1.6e7"),
        # particles kept on the host by the calling program
        dict(_case("host", "fp32", "plummer", 1000000, 16, 0.5, 2), name="host_fp32_plummer_1e6"),
        # a binary on its orbit: kick-drift-kick, the tree rebuilt every step
        dict(_case("leapfrog", "fp64", "binary", 13000, 16, 0.5, 2, nsteps=8), name="leapfrog_fp64_binary_13e3"),
    ]


def draw(rng):
    top = max(_cost(c) for c in listed())
    while True:
        entry = rng.choice(["step", "step", "step", "graph", "host", "leapfrog", "ensemble"])
        form = rng.choice(["fp32", "fp32", "fp64"])
        leaf = rng.choice([8, 10, 12, 16, 20, 24, 32])
        theta = round(rng.uniform(0.3, 0.8), 3)
        order = rng.choice([1, 2, 2, 2, 3, 4])
        if entry == "ensemble":
            c = _case("graph", form, "ensemble", int(round(math.exp(rng.uniform(math.log(2), math.log(300))))), 0, theta, order)
        elif entry == "leapfrog":
            n = int(math.exp(rng.uniform(math.log(1e3), math.log(1e5))))
            c = _case(entry, form, "binary", n, leaf, theta, order, nsteps=rng.randint(2, 8))
        else:
            n = int(math.exp(rng.uniform(math.log(500), math.log(1.6e7))))
            c = _case(entry, form, rng.choice(["uniform", "plummer", "binary", "cloud"]), n, leaf, theta, order)
        if _cost(c) <= top:
            return c


def _counts(case):
    """(particles, near pairs, node-node interactions) of one gravity call,
    from fits to this method's counts over the declared ranges."""
    n, leaf, th = case["n"], case["leaf"], case["theta"]
    sizes = _ensemble_sizes(n) if case["profile"] == "ensemble" else [n]
    pairs = m2l = 0.0
    for s in sizes:
        lf = leaf or _system_leaf(s)
        pairs += s * min(float(s), 110.0 * lf * max(0.6, (0.5 / th) ** 2))
        m2l += s * min(s / 40.0, 27.0 * (16.0 / lf) * (0.5 / th) ** 1.6)
    return sum(sizes), pairs, m2l


def work(case):
    n, pairs, m2l = _counts(case)
    p = case["order"]
    ncoef = (p + 1) * (p + 2) * (p + 3) // 6 + (p + 2) * (p + 3) * (p + 4) // 6 - 1
    calls = case.get("nsteps", 0) + 1
    # 20 operations per softened pair; derivatives and contraction per M2L
    flops = calls * (20.0 * pairs + m2l * ncoef * (p + 2) * 1.2)
    nbytes = 72.0 * n if case["entry"] != "leapfrog" else 112.0 * n
    return {"bytes": nbytes, "flops": flops}


def _cost(case):
    w = work(case)
    return w["flops"] * (26.0 if case["form"] == "fp64" else 1.0) + 300.0 * w["bytes"]


def tolerance(case):
    """Relative errors that summation order and another correct evaluation at
    the same precision show: about four times what was measured against
    ``exact``, which is 0.8e-7 to 3.2e-7 of the result's norm in the FP32 form
    and 0.9e-15 to 2.6e-15 in the FP64 form; single values (a particle where
    the field nearly cancels) up to 100 times the norm's error."""
    if case["form"] == "fp64":
        return {"rel": 1e-14, "max": 1e-12}
    if case["entry"] == "leapfrog":
        return {"rel": 2e-6, "max": 2e-4}
    return {"rel": 1e-6, "max": 1e-4}


# --------------------------------------------------------------------------
# Particle sets (drawn on the device from the seed)
# --------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=_dev())
    g.manual_seed(int(seed))
    return g


def _u(g, n, lo=0.0, hi=1.0):
    return torch.rand(n, generator=g, device=_dev(), dtype=torch.float64) * (hi - lo) + lo


def _directions(g, n):
    mu, phi = _u(g, n, -1.0, 1.0), _u(g, n, 0.0, 2.0 * math.pi)
    s = torch.sqrt(torch.clamp(1.0 - mu * mu, min=0.0))
    return torch.stack([s * torch.cos(phi), s * torch.sin(phi), mu], 1)


def _plummer_radii(g, n, a, rtrunc):
    umax = (rtrunc * rtrunc / (a * a + rtrunc * rtrunc)) ** 1.5
    u = torch.clamp(_u(g, n, 0.0, umax), min=1e-30)
    return a / torch.sqrt(u ** (-2.0 / 3.0) - 1.0)


def _plummer_rho(r2, a, mass):
    return 3.0 * mass * a * a / (4.0 * math.pi * (a * a + r2) ** 2.5)


def _with_h(pos, rho):
    n = pos.shape[0]
    m = torch.full((n,), 1.0 / n, dtype=torch.float64, device=pos.device)
    return pos.contiguous(), m, HFACT * (m / rho) ** (1.0 / 3.0)


def _uniform(g, n):
    pos = (_u(g, n) ** (1.0 / 3.0))[:, None] * _directions(g, n)
    return _with_h(pos, torch.full((n,), 3.0 / (4.0 * math.pi), dtype=torch.float64, device=pos.device))


def _plummer(g, n):
    pos = _plummer_radii(g, n, 1.0, 20.0)[:, None] * _directions(g, n)
    return _with_h(pos, _plummer_rho((pos * pos).sum(1), 1.0, 1.0))


_LE = []


def _lane_emden():
    """n = 1.5 Lane-Emden table (xi, theta, enclosed mass), by RK4."""
    if not _LE:
        f = lambda x, t, d: (d, -max(t, 0.0) ** 1.5 - 2.0 * d / x)  # noqa: E731
        x, k = 1e-3, 1e-3
        t, d = 1.0 - x * x / 6.0, -x / 3.0
        rows = [(0.0, 1.0, 0.0), (x, t, -x * x * d)]
        while t > 0.0:
            a = f(x, t, d)
            b = f(x + k / 2, t + k / 2 * a[0], d + k / 2 * a[1])
            c = f(x + k / 2, t + k / 2 * b[0], d + k / 2 * b[1])
            e = f(x + k, t + k * c[0], d + k * c[1])
            x, t, d = x + k, t + k / 6 * (a[0] + 2 * b[0] + 2 * c[0] + e[0]), d + k / 6 * (a[1] + 2 * b[1] + 2 * c[1] + e[1])
            rows.append((x, max(t, 0.0), -x * x * d))
        _LE.append([torch.tensor(v, dtype=torch.float64, device=_dev()) for v in zip(*rows)])
    return _LE[0]


def _interp(x, xp, fp):
    i = torch.clamp(torch.searchsorted(xp, x, right=True) - 1, 0, xp.numel() - 2)
    w = (x - xp[i]) / (xp[i + 1] - xp[i])
    return fp[i] + w * (fp[i + 1] - fp[i])


def _star(g, n, mass, radius, x0):
    xi, th, mu = _lane_emden()
    rho_c = mass * xi[-1] ** 3 / (4.0 * math.pi * radius ** 3 * mu[-1])
    q = _interp(torch.clamp(_u(g, n), max=1.0 - 0.5 / n) * mu[-1], mu, xi)
    pos = (radius / xi[-1] * q)[:, None] * _directions(g, n)
    pos[:, 0] += x0
    return pos, torch.clamp(rho_c * _interp(q, xi, th) ** 1.5, min=1e-6 * float(rho_c))


def _binary(g, n):
    """Two polytropes, mass ratio 0.3, radii 1 and 0.6, 3 apart on x."""
    m1, m2 = 1.0 / 1.3, 0.3 / 1.3
    n1 = int(round(n * m1))
    (p1, r1), (p2, r2) = _star(g, n1, m1, 1.0, -3.0 * m2), _star(g, n - n1, m2, 0.6, 3.0 * m1)
    return _with_h(torch.cat([p1, p2]), torch.cat([r1, r2]))


def _cloud(g, n):
    """Plummer halo with 70 % of the mass and 64 Plummer clumps (scale 0.02,
    log-normal masses), each clump's density truncated where it ends."""
    nc, a, rcut = 64, 0.02, 0.4
    cm = np.random.default_rng(g.initial_seed() % (1 << 31)).lognormal(0.0, 1.0, nc)
    cm *= 0.3 / cm.sum()
    counts = np.floor(cm * n).astype(np.int64)
    centres = _plummer_radii(g, nc, 1.0, 5.0)[:, None] * _directions(g, nc)
    nh = int(n - counts.sum())
    pos = torch.cat([_plummer_radii(g, nh, 1.0, 20.0)[:, None] * _directions(g, nh)]
                    + [_plummer_radii(g, int(k), a, rcut)[:, None] * _directions(g, int(k)) + centres[c]
                       for c, k in enumerate(counts)])
    rho = _plummer_rho((pos * pos).sum(1), 1.0, 0.7)
    for c in range(nc):
        r2 = ((pos - centres[c]) ** 2).sum(1)
        rho += torch.where(r2 < rcut * rcut, _plummer_rho(r2, a, float(cm[c])), torch.zeros_like(r2))
    return _with_h(pos, rho)


def _ensemble_sizes(nsys):
    """System sizes, log-uniform in [10^3, 10^5]; the same for every seed, as
    a program that runs the same models again has them."""
    return [int(10.0 ** v) for v in np.random.default_rng(1004 + nsys).uniform(3.0, 5.0, nsys)]


def _system_leaf(s):
    return 16 if s >= 20000 else 8


def _ensemble(g, nsys):
    sizes = _ensemble_sizes(nsys)
    parts = [(_plummer if k % 2 == 0 else _uniform)(g, s) for k, s in enumerate(sizes)]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    return [torch.cat([p[k] for p in parts]) for k in range(3)], off, np.array([_system_leaf(s) for s in sizes], np.int32)


def _particles(case, seed):
    return {"uniform": _uniform, "plummer": _plummer, "binary": _binary, "cloud": _cloud}[case["profile"]](_gen(seed), case["n"])


def _orbit(pos):
    """Circular-orbit velocities of the two stars (G M = 1, 3 apart)."""
    n = pos.shape[0]
    n1 = int(round(n / 1.3))
    v = torch.zeros_like(pos)
    v[:n1, 1] = -math.sqrt(1.0 / 3.0) * (n - n1) / n
    v[n1:, 1] = math.sqrt(1.0 / 3.0) * n1 / n
    return v


DT = 2.0 * math.pi * math.sqrt(27.0) / 400.0  # 400 steps per orbit


# --------------------------------------------------------------------------
# The passes
# --------------------------------------------------------------------------
def prepare(case, seed):
    s = dict(case=case, solver=sfmm.Solver(0, case["form"]))
    if case["profile"] == "ensemble":
        (pos, m, h), s["off"], s["leaf"] = _ensemble(_gen(seed), case["n"])
    else:
        pos, m, h = _particles(case, seed)
        s["off"], s["leaf"] = np.array([0, case["n"]], np.int64), np.array([case["leaf"]], np.int32)
    if case["entry"] == "host":
        pos, m, h = (t.cpu().pin_memory() for t in (pos, m, h))
        s["acc"], s["pot"] = torch.empty_like(pos).pin_memory(), torch.empty_like(m).pin_memory()
    elif case["entry"] == "graph":
        s["acc"], s["pot"] = torch.empty_like(pos), torch.empty_like(m)
    elif case["entry"] == "leapfrog":
        s["vel"] = _orbit(pos)
    s["pos"], s["m"], s["h"] = pos, m, h
    return s


def run(s):
    c, solver = s["case"], s["solver"]
    if c["entry"] == "step":
        solver.build(s["pos"], s["m"], s["h"], c["leaf"])
        acc, pot = solver.gravity(c["theta"], c["order"])
        return {"acc": acc, "pot": pot}
    if c["entry"] == "graph":
        sfmm.sfmm_solve_graph(solver.ctx, s["off"], s["pos"], s["m"], s["h"], s["leaf"], c["theta"], c["order"], s["acc"], s["pot"])
        return {"acc": s["acc"], "pot": s["pot"]}
    if c["entry"] == "host":
        solver.solve_host(s["pos"], s["m"], s["h"], c["leaf"], c["theta"], c["order"], s["acc"], s["pot"])
        return {"acc": s["acc"], "pot": s["pot"]}
    pos, vel, rec = solver.leapfrog(s["pos"], s["vel"], s["m"], s["h"], c["leaf"], c["theta"], c["order"], DT, c["nsteps"])
    return {"pos": pos, "vel": vel, "records": rec}


# --------------------------------------------------------------------------
# The same in float64, in plain torch
# --------------------------------------------------------------------------
def exact(case, seed):
    n, pairs, m2l = _counts(case)
    if (pairs + 30.0 * m2l) * (case.get("nsteps", 0) + 1) > 1.2e10:
        return None  # over about 20 seconds
    p = case["order"]
    if case["profile"] == "ensemble":
        (pos, m, h), off, leaf = _ensemble(_gen(seed), case["n"])
        got = [_sfmm(pos[a:b], m[a:b], h[a:b], int(k), case["theta"], p) for a, b, k in zip(off[:-1], off[1:], leaf)]
        return {"acc": torch.cat([g[0] for g in got]), "pot": torch.cat([g[1] for g in got])}
    pos, m, h = _particles(case, seed)
    if case["entry"] != "leapfrog":
        acc, pot = _sfmm(pos, m, h, case["leaf"], case["theta"], p)
        if case["entry"] == "host":
            acc, pot = acc.cpu(), pot.cpu()
        return {"acc": acc, "pot": pot}
    vel = _orbit(pos)
    rec = []

    def note(t):
        mv = m[:, None] * vel
        rec.append([t] + mv.sum(0).tolist() + torch.linalg.cross(pos, mv).sum(0).tolist() + [float(mv.abs().sum())])

    note(0.0)
    acc, _ = _sfmm(pos, m, h, case["leaf"], case["theta"], p)
    for k in range(case["nsteps"]):
        vel = vel + acc * (0.5 * DT)
        pos = pos + vel * DT
        acc, _ = _sfmm(pos, m, h, case["leaf"], case["theta"], p)
        vel = vel + acc * (0.5 * DT)
        note((k + 1) * DT)
    return {"pos": pos, "vel": vel, "records": np.array(rec)}


def _multi_indices(k, lo=0):
    return [(a, b, d - a - b) for d in range(lo, k + 1) for a in range(d, -1, -1) for b in range(d - a, -1, -1)]


def _plus(a, b):
    return tuple(x + y for x, y in zip(a, b))


def _monomials(v, k):
    """v^alpha / alpha! for |alpha| <= k, as a dict of vectors."""
    out = {(0, 0, 0): torch.ones_like(v[:, 0])}
    for g in _multi_indices(k, 1):
        t = next(i for i in range(3) if g[i])
        out[g] = out[tuple(x - (i == t) for i, x in enumerate(g))] * v[:, t] / g[t]
    return out


def _derivatives(r, k):
    """D_gamma = d^gamma (1 / |r|) for |gamma| <= k (McMurchie-Davidson)."""
    rinv2 = 1.0 / (r * r).sum(1)
    base = [torch.sqrt(rinv2)]
    for j in range(k):
        base.append(base[-1] * rinv2 * -(2 * j + 1))
    have = {}

    def get(j, g):
        if g == (0, 0, 0):
            return base[j]
        if (j, g) not in have:
            t = next(i for i in range(3) if g[i])
            v = r[:, t] * get(j + 1, tuple(x - (i == t) for i, x in enumerate(g)))
            if g[t] > 1:
                v = v + (g[t] - 1) * get(j + 1, tuple(x - 2 * (i == t) for i, x in enumerate(g)))
            have[(j, g)] = v
        return have[(j, g)]

    return {g: get(0, g) for g in _multi_indices(k)}


def _spread(v):
    """21 bits, two zero bits after each."""
    for s, mask in ((32, 0x1F00000000FFFF), (16, 0x1F0000FF0000FF), (8, 0x100F00F00F00F00F), (4, 0x10C30C30C30C30C3),
                    (2, 0x1249249249249249)):
        v = (v | (v << s)) & mask
    return v


def _highest_bit(v):
    """Position of the highest set bit of each v > 0 (below 2^63)."""
    b = torch.zeros_like(v)
    for s in (32, 16, 8, 4, 2, 1):
        up = (v >> s) > 0
        b, v = torch.where(up, b + s, b), torch.where(up, v >> s, v)
    return b


def _tree(pos, leaf):
    """Radix tree over Morton keys, nodes in breadth-first order: sorted
    order of the particles, first, count, children, parent, levels."""
    n, dev = pos.shape[0], pos.device
    lo = pos.min(0).values
    extent = float((pos.max(0).values - lo).max())
    q = torch.clamp(torch.floor((pos - lo) * ((2.0 ** 21) / extent if extent > 0 else 0.0)), 0, 2 ** 21 - 1).to(torch.int64)
    key = (_spread(q[:, 0]) << 2) | (_spread(q[:, 1]) << 1) | _spread(q[:, 2])
    key, order = torch.sort(key, stable=True)
    first, last = [torch.zeros(1, dtype=torch.int64, device=dev)], [torch.full((1,), n - 1, dtype=torch.int64, device=dev)]
    parent, left, levels, base = [torch.full((1,), -1, dtype=torch.int64, device=dev)], [], [(0, 1)], 0
    while True:
        f, l = first[-1], last[-1]
        split = (l - f + 1) > leaf
        lc = torch.full_like(f, -1)
        at = torch.nonzero(split).flatten()
        base += f.numel()
        lc[at] = base + 2 * torch.arange(at.numel(), device=dev)
        left.append(lc)
        if not at.numel():
            break
        f, l = f[at], l[at]
        kf, kl = key[f], key[l]
        same = kf == kl
        x = torch.where(same, f ^ l, kf ^ kl)
        b = _highest_bit(x)
        cut = torch.where(same, (l >> b) << b, torch.searchsorted(key, (kl >> b) << b))
        first.append(torch.stack([f, cut], 1).flatten())
        last.append(torch.stack([cut - 1, l], 1).flatten())
        parent.append((base - split.numel() + at).repeat_interleave(2))
        levels.append((base, base + 2 * at.numel()))
    first, last, left, parent = (torch.cat(v) for v in (first, last, left, parent))
    return order, first, last - first + 1, left, parent, levels


def _sfmm(pos_in, m_in, h_in, leaf_size, theta, p):
    """Accelerations and potentials (G = 1, no self term), caller order."""
    dev, n = pos_in.device, pos_in.shape[0]
    order, first, count, left, parent, levels = _tree(pos_in, leaf_size)
    pos, m, h = pos_in[order], m_in[order], h_in[order]
    nn = first.numel()
    zeros = lambda *s: torch.zeros(*s, dtype=torch.float64, device=dev)  # noqa: E731
    leaves = torch.nonzero(left < 0).flatten()
    by_first = leaves[torch.argsort(first[leaves])]
    pleaf = by_first.repeat_interleave(count[by_first])  # leaf of each particle

    # masses, centres, largest h: particles to leaves, then level by level
    mass, mx, hmax = zeros(nn).index_add(0, pleaf, m), zeros(nn, 3).index_add(0, pleaf, m[:, None] * pos), zeros(nn)
    hmax = hmax.scatter_reduce(0, pleaf, h, "amax")
    for a, b in levels[:0:-1]:
        up = parent[a:b]
        mass.index_add_(0, up, mass[a:b].clone())
        mx.index_add_(0, up, mx[a:b].clone())
        hmax.scatter_reduce_(0, up, hmax[a:b].clone(), "amax")
    cen = mx / mass[:, None]
    # sizes: the largest distance of a node's particles from its centre
    size, node, live = zeros(nn), pleaf, torch.arange(n, device=dev)
    while live.numel():
        size.scatter_reduce_(0, node, ((pos[live] - cen[node]) ** 2).sum(1).sqrt(), "amax")
        node = parent[node]
        live, node = live[node >= 0], node[node >= 0]
    # scaled moments Q_alpha / alpha! about the centres
    mi = _multi_indices(p)
    mono = _monomials(pos - cen[pleaf], p)
    Q = {a: zeros(nn).index_add(0, pleaf, m * mono[a]) for a in mi}
    for a, b in levels[:0:-1]:
        up = parent[a:b]
        sh = _monomials(cen[a:b] - cen[up], p)
        for al in reversed(mi):
            v = sum(sh[tuple(x - y for x, y in zip(al, be))] * Q[be][a:b] for be in mi if all(x >= y for x, y in zip(al, be)))
            Q[al].index_add_(0, up, v)

    # dual-tree walk from (root, root); targets keep their sums
    mf = _multi_indices(p + 1, 1)
    M, F = {b: zeros(nn) for b in mi}, {g: zeros(nn) for g in mf}

    def m2l(A, S):
        D = _derivatives(cen[S] - cen[A], p + 1)
        q = {a: Q[a][S] for a in mi}
        for out, idx, top in ((M, mi, p), (F, mf, p + 1)):
            for g in idx:
                v = sum(D[_plus(a, g)] * q[a] for a in mi if sum(a) <= top - sum(g))
                out[g].index_add_(0, A, v if sum(g) % 2 == 0 else -v)

    near = []
    todo = [(torch.zeros(1, dtype=torch.int64, device=dev), torch.zeros(1, dtype=torch.int64, device=dev))]
    while todo:
        A, S = todo.pop()
        if A.numel() > 1 << 23:
            todo += [(A[1 << 23:], S[1 << 23:])]
            A, S = A[:1 << 23], S[:1 << 23]
        d = ((cen[S] - cen[A]) ** 2).sum(1).sqrt()
        ls = size[A] + size[S]
        ok = (A != S) & (ls < theta * d) & ~(d < ls + 2.0 * torch.maximum(hmax[A], hmax[S]))
        acc_at = torch.nonzero(ok).flatten()
        for c in acc_at.split(1 << 21):
            m2l(A[c], S[c])
        A, S = A[~ok], S[~ok]
        la, ls_ = left[A] < 0, left[S] < 0
        both = la & ls_
        if bool(both.any()):
            near.append((A[both], S[both]))
        nxt = []
        k = ~la & ~ls_
        nxt += [(left[A[k]] + i, left[S[k]] + j) for i in (0, 1) for j in (0, 1)]
        k = ~la & ls_
        nxt += [(left[A[k]] + i, S[k]) for i in (0, 1)]
        k = la & ~ls_
        nxt += [(A[k], left[S[k]] + j) for j in (0, 1)]
        A, S = torch.cat([x[0] for x in nxt]), torch.cat([x[1] for x in nxt])
        if A.numel():
            todo.append((A, S))

    # coefficients down the tree, then evaluated at the particles
    for a, b in levels[1:]:
        up = parent[a:b]
        sh = _monomials(cen[a:b] - cen[up], p + 1)
        for C, idx in ((M, mi), (F, mf)):
            for g in idx:
                C[g][a:b] += sum(sh[tuple(x - y for x, y in zip(k, g))] * C[k][up] for k in idx if all(x >= y for x, y in zip(k, g)))
    acc = torch.stack([sum(mono[b] * F[_plus(b, e)][pleaf] for b in mi) for e in ((1, 0, 0), (0, 1, 0), (0, 0, 1))], 1)
    pot = -sum(mono[b] * M[b][pleaf] for b in mi)

    # softened pairs of the leaf-leaf list
    A, S = (torch.cat([x[k] for x in near]) for k in (0, 1)) if near else (leaves[:0], leaves[:0])
    size_of = count[A] * count[S]
    ends = torch.cumsum(size_of, 0)
    at, total, step = 0, int(ends[-1]) if A.numel() else 0, 1 << 24
    while at < A.numel():
        to = max(at + 1, int(torch.searchsorted(ends, (int(ends[at - 1]) if at else 0) + step)))
        a, s, k = A[at:to], S[at:to], size_of[at:to]
        pair = torch.arange(to - at, device=dev).repeat_interleave(k)
        o = torch.arange(pair.numel(), device=dev) - (torch.cumsum(k, 0) - k)[pair]
        ns = count[s][pair]
        i, j = first[a][pair] + o // ns, first[s][pair] + o % ns
        keep = i != j
        i, j = i[keep], j[keep]
        d = pos[i] - pos[j]
        r = (d * d).sum(1).sqrt()
        g, phi = torch.zeros_like(r), torch.zeros_like(r)
        for hh in (h[i], h[j]):
            gk, pk = _m4(r, hh)
            g += 0.5 * gk
            phi += 0.5 * pk
        acc.index_add_(0, i, -(m[j] * g)[:, None] * d)
        pot.index_add_(0, i, m[j] * phi)
        at = to
    out_a, out_p = torch.empty_like(acc), torch.empty_like(pot)
    out_a[order], out_p[order] = acc, pot
    return out_a, out_p


def _m4(r, h):
    """phi'(r) / r and phi(r) of a unit mass in the M4 kernel of length h."""
    q = r / h
    rs = torch.clamp(r, min=1e-300)
    g = torch.where(q < 1.0, (4.0 / 3.0 - 1.2 * q ** 2 + 0.5 * q ** 3) / h ** 3,
                    (8.0 / 3.0 - 3.0 * q + 1.2 * q ** 2 - q ** 3 / 6.0) / h ** 3 - 1.0 / (15.0 * rs ** 3))
    f = torch.where(q < 1.0, (-1.4 + 2.0 / 3.0 * q ** 2 - 0.3 * q ** 4 + 0.1 * q ** 5) / h,
                    (-1.6 + 4.0 / 3.0 * q ** 2 - q ** 3 + 0.3 * q ** 4 - q ** 5 / 30.0) / h + 1.0 / (15.0 * rs))
    out = q >= 2.0
    return torch.where(out, 1.0 / rs ** 3, g), torch.where(out, -1.0 / rs, f)
