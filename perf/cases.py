"""The work that programs have this framework do, as cases that can be measured.

A case is one call sequence of a user's program through the public entry
points of paper_1907_02289_gb300.bh, on seeded synthetic particles that are
drawn on the GPU:

  evaluate    bh_build_tree, bh_make_lists, bh_compute_forces: a whole
              list-constructing force evaluation (tree part)
  forces      bh_compute_forces on lists that stand: a list-reusing evaluation
  steps       bh_step of 4 leapfrog steps on device arrays: one whole cycle of
              the list-reuse schedule, with one list build in it
  host_steps  the same through bh_step_host on page-locked host arrays
  energy      bh_get_diagnostics and bh_compute_potential on lists that stand
  sort        bh_sort_keys_static on Morton keys of a ring's particles

Particles: "ring" is the whole annulus and "patches" independent sectors of
one (the recipe of paper_1907_02289_gb300.synth: r uniform in [0.98, 1.02], z
Gaussian of 1e-4, Kepler velocities with a dispersion of 1e-4, mass 1e-12,
contacts at 2e-5 with the spring and dashpot of synth.contact_params); "cube"
is the uniform unit cube at rest with softening 1e-3.
"""
import math

import numpy as np
import torch

from paper_1907_02289_gb300 import bh, synth

TWO_PI = 2.0 * math.pi
MASS, SURFACE_N = 1e-12, 1 << 20  # ring particle; the patches' surface density is that of a ring of so many
STEPS, DT = 4, synth.DT
ALL = ("x", "y", "z", "vx", "vy", "vz", "m", "id", "ax", "ay", "az")


def _case(name, op, shape, n, **kw):
    """A case with every option stated.  patches, size_seed: how many patches
    and the seed of their sizes; warps: warps per block of the FP32 kernel."""
    c = dict(op=op, shape=shape, n=n, patches=1, size_seed=0, theta=0.5, n_g=128, order=2, precision=1, frame=0,
             omega=0.0, graph=0, warps=4)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the uniform cube's force evaluation, FP64, softened, monopole: 4096
        # particles, where launches, waits and idle SMs count
        _case("evaluate_cube_4096_f64", "evaluate", "cube", 4096, n_g=64, order=1, precision=0),
        # one list-reusing evaluation of a small ring: the smallest call of a
        # program that keeps its lists
        _case("forces_ring_20000", "forces", "ring", 20000, n_g=64),
        # an ordinary ring of odd size, evaluated from its particles to its
        # forces each time (a program that moves the particles itself)
        _case("evaluate_ring_65537", "evaluate", "ring", 65537),
        # a softened cloud, monopole only, FP32: no contacts, no quadrupole
        _case("evaluate_cube_100003", "evaluate", "cube", 100003, theta=0.6, n_g=64, order=1),
        # time stepping of a small ring in the rotating frame, with the
        # cylindrical tree and every step a CUDA graph
        _case("steps_ring_300007_graph", "steps", "ring", 300007, frame=1, omega=1.0, graph=1, warps=8),
        # the energies that a simulation prints beside its steps
        _case("energy_ring_262144", "energy", "ring", 262144),
        # the plain FP64 path's time stepping: the 2^20 ring
        _case("steps_ring_2p20_f64", "steps", "ring", 1 << 20, precision=0),
        # a program whose particles live in host memory between calls
        _case("host_steps_ring_2p20", "host_steps", "ring", 1 << 20, frame=1),
        # many independent patches of uneven size in one context, in graphs,
        # with the launch settings that the autotuner picks for them
        _case("steps_patches_64", "steps", "patches", int(synth.patch_sizes(64, 3).sum()), patches=64, size_seed=3,
              n_g=96, graph=1, warps=8),
        # the 2^24 ring, FP32 forces
        _case("steps_ring_2p24", "steps", "ring", 1 << 24),
        # the large ring of the benchmark, with its autotuned settings
        _case("steps_ring_2p26", "steps", "ring", 1 << 26, theta=0.4, n_g=192, frame=1, warps=8),
        # the key sort on its own, on the caller's buffers
        _case("sort_keys_3000001", "sort", "ring", 3000001),
    ]


def draw(rng):
    """One more case of the same ranges, sizes log-uniform."""
    op = rng.choice(("evaluate", "forces", "steps", "steps", "energy", "sort", "host_steps"))

    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    if op == "sort":
        return _case("", op, "ring", size(1000, bh.BH_SORT_STATIC_MAX_N))
    kw = dict(theta=round(rng.uniform(0.4, 0.8), 3), n_g=rng.choice((32, 64, 96, 128, 192, 256)),
              order=rng.choice((1, 2, 2)), precision=rng.choice((0, 1, 1)), warps=rng.choice((4, 8)))
    shape = rng.choice(("ring", "ring", "cube", "patches"))
    if op in ("steps", "host_steps") and shape == "cube":
        shape = "ring"  # the cloud at rest is evaluated, not stepped
    if op == "host_steps" and shape == "patches":
        shape = "ring"
    big = (1 << 18 if shape == "cube" else 1 << 19) if kw["precision"] == 0 or op == "energy" else 1 << 22
    if op == "host_steps":
        big = min(big, 1 << 21)
    if shape != "cube":
        kw["frame"] = rng.choice((0, 1))
    if op == "steps":
        kw.update(graph=rng.choice((0, 1)), omega=rng.choice((0.0, 1.0)))
    if shape == "patches":
        kw.update(patches=rng.randint(2, 64), size_seed=rng.randrange(1 << 20))
        n = int(_sizes(kw["patches"], kw["size_seed"], size(2000, big)).sum())
        return _case("", op, shape, n, **kw)
    return _case("", op, shape, size(1000, big), **kw)


def _sizes(patches, size_seed, total):
    """Uneven patch sizes (log-uniform over a factor of 50) of about `total`."""
    w = np.exp(np.random.default_rng(size_seed).uniform(0.0, math.log(50.0), patches))
    return np.maximum(1, np.rint(w * (total / w.sum()))).astype(np.int64)


def _offsets(c):
    if c["patches"] == 1:
        return [0, c["n"]]
    if (c["patches"], c["size_seed"]) == (64, 3):
        s = synth.patch_sizes(64, 3)
    else:
        s = _sizes(c["patches"], c["size_seed"], c["n"])
        s[-1] += c["n"] - s.sum()  # (the rounded sizes of the rounded total)
    return [0] + [int(v) for v in np.cumsum(s)]


def _params(c):
    kappa, eta = synth.contact_params(DT)
    ring = c["shape"] != "cube"
    return dict(theta=c["theta"], eps=0.0 if ring else 1e-3, G=1.0, M_central=1.0 if ring else 0.0,
                r_coll=2 * synth.PARTICLE_RADIUS if ring else 0.0, kappa=kappa if ring else 0.0,
                eta=eta if ring else 0.0, dt=DT, n_g=c["n_g"], n_leaf=8, order=c["order"], precision=c["precision"],
                rebuild_every=STEPS, key_frame=c["frame"], omega=c["omega"])


def _particles(c, seed, dev="cuda"):
    """x .. vz, m, id of the case, on the device."""
    n = c["n"]
    g = torch.Generator(device=dev).manual_seed(int(seed) * 7919 + 13)

    def uniform(lo, hi):
        return torch.rand(n, generator=g, device=dev, dtype=torch.float64) * (hi - lo) + lo

    def normal(s):
        return torch.randn(n, generator=g, device=dev, dtype=torch.float64) * s

    P = {"id": torch.arange(n, device=dev)}
    if c["shape"] == "cube":
        P.update(x=uniform(0, 1), y=uniform(0, 1), z=uniform(0, 1), m=torch.full((n,), 1.0 / n, device=dev).double())
        for f in ("vx", "vy", "vz"):
            P[f] = torch.zeros(n, device=dev, dtype=torch.float64)
        return P
    r, phi = uniform(0.98, 1.02), uniform(0.0, TWO_PI)
    if c["shape"] == "patches":  # each a sector of its own size
        off = _offsets(c)
        for a, b in zip(off[:-1], off[1:]):
            phi[a:b] *= (b - a) / SURFACE_N
    vk, co, si = r.rsqrt(), phi.cos(), phi.sin()
    P.update(x=r * co, y=r * si, z=normal(1e-4), m=torch.full((n,), MASS, device=dev, dtype=torch.float64))
    P.update(vx=normal(1e-4) - vk * si, vy=normal(1e-4) + vk * co, vz=normal(1e-4))
    return P


def prepare(case, seed):
    c = case
    P = _particles(c, seed)
    if c["op"] == "sort":
        key, _ = _keys(P, _params(c))
        return dict(c=c, src=key[torch.randperm(c["n"], device="cuda", generator=torch.Generator("cuda").manual_seed(int(seed)))],
                    key=torch.empty_like(key), ktmp=torch.empty_like(key),
                    idx=torch.empty(c["n"], dtype=torch.int32, device="cuda"),
                    itmp=torch.empty(c["n"], dtype=torch.int32, device="cuda"))
    ctx = bh.Context(offsets=_offsets(c) if c["patches"] > 1 else None, **_params(c))
    ctx.bh_set_tuning(warps=c["warps"], graph=c["graph"])
    s = dict(c=c, ctx=ctx)
    if c["op"] == "host_steps":
        s["D"] = bh.HostParticles({f: v.cpu().numpy() for f, v in P.items()}, pinned=True)
        ctx.bh_step_host(s["D"], 0)  # the initial acceleration, and the first lists
        return s
    D = s["D"] = bh.Particles({"x": np.zeros(c["n"])})
    for f, v in P.items():
        D.t[f].copy_(v)
    if c["op"] == "steps":
        ctx.bh_step(D, 0)
    elif c["op"] in ("forces", "energy"):
        ctx.bh_build_tree(D)
        ctx.bh_make_lists()
    if c["op"] == "energy":
        s["phi"] = torch.empty(c["n"], dtype=torch.float64, device="cuda")
    return s


def run(state):
    s = state
    op = s["c"]["op"]
    if op == "sort":
        s["key"].copy_(s["src"])
        bh.bh_sort_keys_static(s["key"], s["idx"], s["ktmp"], s["itmp"])
        return {"key": s["key"], "idx": s["idx"]}
    ctx, D = s["ctx"], s["D"]
    if op == "evaluate":
        ctx.bh_build_tree(D)
        ctx.bh_make_lists()
        ctx.bh_compute_forces(D, bh.BH_FORCE_TREE_ONLY)
        return {f: D.t[f] for f in ALL}
    if op == "forces":
        ctx.bh_compute_forces(D, bh.BH_FORCE_TREE_ONLY)
        return {f: D.t[f] for f in ("ax", "ay", "az")}
    if op == "steps":
        ctx.bh_step(D, STEPS)
        return {f: D.t[f] for f in ALL}
    if op == "host_steps":
        ctx.bh_step_host(D, STEPS)
        return {f: D.a[f] for f in ALL}
    d = ctx.bh_get_diagnostics(D)
    W = ctx.bh_compute_potential(D, s["phi"])
    return {"phi": s["phi"], "W": W, "mass": d["mass"], "kinetic": d["kinetic"], "central": d["potential_central"],
            "momentum": d["momentum"], "angular_momentum": d["angular_momentum"]}


def _interactions(c):
    """About how many list particles and list cells a particle meets (counted
    with the CPU oracle on rings of 5,000 to 2^26 particles and cubes of 1,000
    to 300,000; within a third or so)."""
    n = c["n"] if c["patches"] == 1 else SURFACE_N
    w = 0.5 / c["theta"]
    if c["shape"] == "cube":
        return 7.0 * c["n_g"] * w ** 2, 200.0 * max(1.0, math.log2(n) - 9.0) * w ** 2
    return (1.6 * c["n_g"] + 60.0) * w ** 2, 33.0 * max(1.0, math.log2(n) - 11.5) * w ** 3


def work(case):
    """Bytes: the particle arrays that the call reads, in, and those that it
    changes, out (for each of several steps: a force needs every particle's
    new position).  Flops: the lists' interactions, 23 per list particle and 48
    (quadrupole) or 18 per list cell."""
    c = case
    n = c["n"]
    if c["op"] == "sort":
        return {"bytes": 20.0 * n, "flops": 0.0}
    pp, pc = _interactions(c)
    flops = n * (23.0 * pp + (48.0 if c["order"] == 2 else 18.0) * pc)
    if c["op"] == "evaluate":
        return {"bytes": n * (64.0 + 88.0), "flops": flops}
    if c["op"] == "forces":
        return {"bytes": n * 56.0, "flops": flops}
    if c["op"] == "energy":
        return {"bytes": n * 64.0, "flops": flops * 0.6}
    return {"bytes": n * STEPS * (80.0 + 72.0), "flops": STEPS * flops}


def tolerance(case):
    """FP64 sums differ by about 1e-15 of the result in another order, and the
    FP32 path's tree accelerations by about 2e-7 of their root mean square
    (its gate is 1e-5 of each value).  After steps the acceleration holds the
    central mass's too, of which that is a small part (1e-8 in z), and the
    positions and velocities carry it times dt.  Permuted arrays may differ
    where a last bit moves a particle over the edge of its key cell."""
    c = case
    if c["op"] == "sort":
        return "exact"
    if c["op"] == "energy":
        return {"rel": 1e-11, "max": 1e-9}
    if c["precision"] == 0:
        return {"rel": 1e-11, "max": 1e-9, "differ": 1e-5}
    if c["op"] in ("steps", "host_steps"):
        return {"rel": 1e-7, "max": 2e-5, "differ": 1e-5}
    return {"rel": 1e-6, "max": 2e-5, "differ": 1e-5}


# ---- the same results from their definitions, in plain torch, 64 bits ------
LEVELS = 21


def _keys(P, prm):
    """Morton keys and grid coordinates of one particle set, and its grid."""
    co = [P["x"], P["y"], P["z"]]
    if prm["key_frame"] == 1:  # (phi, r, z), phi and r as FP32 numbers
        X, Y = co[0].float(), co[1].float()
        ax, ay = X.abs(), Y.abs()
        mx, mn = torch.where(ax > ay, ax, ay), torch.where(ax > ay, ay, ax)
        t = mn / mx

        def f32(v):
            return torch.tensor(v, dtype=torch.float32, device=t.device)

        s3 = f32(1.7320508075688772)
        far = t > f32(0.2679491924311227)
        u = torch.where(far, (t * s3 - 1.0) / (t + s3), t)
        u2 = u * u
        p = f32(-1.0 / 11.0)
        for v in (1.0 / 9.0, -1.0 / 7.0, 1.0 / 5.0, -1.0 / 3.0, 1.0):
            p = p * u2 + f32(v)
        a = torch.where(far, f32(0.5235987755982988), f32(0.0)) + u * p
        a = torch.where(ay > ax, f32(1.5707963267948966) - a, a)
        a = torch.where(X < 0, f32(3.141592653589793) - a, a)
        a = torch.where(Y < 0, f32(6.283185307179586) - a, a)
        co = [a.double(), (X * X + Y * Y).sqrt().double(), co[2]]
    lo = [float(v.min()) for v in co]
    L = max(float(v.max()) - b for v, b in zip(co, lo)) or 1.0
    S = 2097152.0 / L
    q = torch.stack([((v - b) * S).floor().clamp(0, (1 << LEVELS) - 1).long() for v, b in zip(co, lo)])
    key = torch.zeros_like(q[0])
    for b in range(LEVELS):
        for a in range(3):
            key |= ((q[a] >> b) & 1) << (3 * b + 2 - a)
    return key, (q, lo, S)


def _ramp(start, cnt):
    """start[k], start[k] + 1, ... (cnt[k] values) for every k, and k itself."""
    k = torch.repeat_interleave(torch.arange(len(cnt), device=cnt.device), cnt)
    return torch.arange(len(k), device=cnt.device) - (torch.cumsum(cnt, 0) - cnt)[k] + start[k], k


def _build(P, prm):
    """Sorted particles, nodes, groups and lists of one particle set."""
    key, (q, lo, S) = _keys(P, prm)
    key, order = torch.sort(key, stable=True)
    P = {f: v[order] for f, v in P.items()}
    q = q[:, order]
    n, dev = len(key), key.device
    one = torch.ones(1, dtype=torch.long, device=dev)
    begin, end, parent, base, levels = [one * 0], [one * n], [one * -1], 0, [(0, 1)]
    first, nchild = [one * -1], [one * 0]
    for l in range(LEVELS):  # children of the nodes of level l
        b, e = begin[-1], end[-1]
        big = torch.nonzero(e - b > prm["n_leaf"]).squeeze(1)
        if not len(big):
            break
        pre = key >> (3 * (LEVELS - 1 - l))
        cut = torch.cat([one * 0, torch.nonzero(pre[1:] != pre[:-1]).squeeze(1) + 1, one * n])
        i0, i1 = torch.searchsorted(cut, b[big]), torch.searchsorted(cut, e[big])
        at, k = _ramp(i0, i1 - i0)
        nxt = base + len(b)
        first[-1][big] = nxt + torch.cumsum(i1 - i0, 0) - (i1 - i0)
        nchild[-1][big] = i1 - i0
        parent.append(base + big[k])
        begin.append(cut[at])
        end.append(cut[at + 1])
        first.append(torch.full_like(at, -1))
        nchild.append(torch.zeros_like(at))
        base = nxt
        levels.append((base, base + len(at)))
    T = dict(prm=prm, P=P, n=n, levels=levels)
    T["begin"], T["end"], T["parent"] = torch.cat(begin), torch.cat(end), torch.cat(parent)
    T["first"], T["nchild"] = torch.cat(first), torch.cat(nchild)
    cnt = T["end"] - T["begin"]
    leaf = torch.nonzero(T["nchild"] == 0).squeeze(1)
    leaf = leaf[torch.argsort(T["begin"][leaf])]
    T["leaf_of"] = torch.repeat_interleave(leaf, cnt[leaf])
    nn = len(cnt)
    qlo, qhi = torch.full((3, nn), 1 << 30, device=dev), torch.full((3, nn), -1, device=dev)
    for a in range(3):
        qlo[a].scatter_reduce_(0, T["leaf_of"], q[a], "amin")
        qhi[a].scatter_reduce_(0, T["leaf_of"], q[a], "amax")
        for s, e in reversed(levels[1:]):
            qlo[a].scatter_reduce_(0, T["parent"][s:e], qlo[a, s:e].clone(), "amin")
            qhi[a].scatter_reduce_(0, T["parent"][s:e], qhi[a, s:e].clone(), "amax")
    # groups: the largest nodes of at most n_g particles
    top = torch.where(T["parent"] < 0, torch.full_like(cnt, 1 << 40), cnt[T["parent"].clamp(min=0)]) > prm["n_g"]
    grp = torch.nonzero(((cnt <= prm["n_g"]) | (T["nchild"] == 0)) & top).squeeze(1)
    grp = T["grp"] = grp[torch.argsort(T["begin"][grp])]
    T["gb"], T["gn"] = T["begin"][grp], cnt[grp]
    # the walk, all groups at once, level by level
    reach, period = prm["r_coll"] * S, 0
    if prm["key_frame"] == 1:
        reach, period = (prm["r_coll"] / lo[1] + 4e-6) * S, math.floor(TWO_PI * S)
    th2, rcq = prm["theta"] ** 2, reach * reach
    pp, pc = [], []
    for at in torch.arange(len(grp), device=dev).split(1 << 16):
        g, node = at, torch.zeros_like(at)
        for l in range(len(levels)):
            d2 = 0
            for a in range(3):
                t1 = qlo[a, node] - qhi[a, grp[g]] - 1
                t2 = qlo[a, grp[g]] - qhi[a, node] - 1
                d = torch.maximum(t1, t2).clamp(min=0)
                if a == 0 and period:
                    round_ = torch.where(t1 > 0, qlo[a, grp[g]] + period - qhi[a, node] - 1,
                                         qlo[a, node] + period - qhi[a, grp[g]] - 1).clamp(min=0)
                    d = torch.where(d > 0, torch.minimum(d, round_), d)
                d2 = d2 + d * d
            d2 = d2.double()
            opened = (th2 * d2 < 4.0 ** (LEVELS - l)) | (d2 <= rcq)
            isleaf = T["nchild"][node] == 0
            pc.append((g[~opened], node[~opened]))
            pp.append((g[opened & isleaf], node[opened & isleaf]))
            g, node = g[opened & ~isleaf], node[opened & ~isleaf]
            kid, k = _ramp(T["first"][node], T["nchild"][node])
            g, node = g[k], kid
    T["pp"] = [torch.cat(v) for v in zip(*pp)]
    T["pc"] = [torch.cat(v) for v in zip(*pc)]
    return T


def _moments(T):
    """Mass, centre and traceless quadrupole of every node."""
    P, nn = T["P"], len(T["begin"])
    xyz = torch.stack([P["x"], P["y"], P["z"]])

    def up(to, frm, m, c, M, cen, Q, q):
        """Add bodies of mass m at c (quadrupole q) to the nodes `to`."""
        d = c - cen[:, to]
        d2 = (d * d).sum(0)
        for k, (a, b) in enumerate(((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))):
            Q[k].index_add_(0, to, m * (3 * d[a] * d[b] - (d2 if a == b else 0.0)) + (q[k] if q is not None else 0.0))

    M = xyz.new_zeros(nn)
    cen, Q = xyz.new_zeros(3, nn), xyz.new_zeros(6, nn)
    M.index_add_(0, T["leaf_of"], P["m"])
    for a in range(3):
        cen[a].index_add_(0, T["leaf_of"], P["m"] * xyz[a])
    isleaf = T["nchild"] == 0
    cen[:, isleaf] /= M[isleaf]
    up(T["leaf_of"], None, P["m"], xyz, M, cen, Q, None)
    for l in range(len(T["levels"]) - 1, 0, -1):
        s, e = T["levels"][l]
        to = T["parent"][s:e]
        M.index_add_(0, to, M[s:e].clone())
        for a in range(3):
            cen[a].index_add_(0, to, (M * cen[a])[s:e])
        u = torch.unique(to)
        cen[:, u] /= M[u]
        up(to, None, M[s:e], cen[:, s:e], M, cen, Q, Q[:, s:e].clone())
    return M, cen, Q


def _pairs(T, which, most=1 << 25):
    """(particle, node) pairs of the lists, in bites of about `most` pairs
    (times the leaf size for list particles)."""
    g, node = T[which]
    per = T["gn"][g] * ((T["end"] - T["begin"])[node] if which == "pp" else 1)
    run_, at = torch.cumsum(per, 0), 0
    while at < len(g):
        done = int(run_[at - 1]) if at else 0
        to = max(at + 1, int(torch.searchsorted(run_, done + most)))
        i, k = _ramp(T["gb"][g[at:to]], T["gn"][g[at:to]])
        nd = node[at:to][k]
        if which == "pp":
            j, k = _ramp(T["begin"][nd], (T["end"] - T["begin"])[nd])
            yield i[k], j
        else:
            yield i, nd
        at = to


def _accelerations(T, central):
    P, prm = T["P"], T["prm"]
    M, cen, Q = _moments(T)
    X = [P["x"], P["y"], P["z"]]
    acc = [torch.zeros_like(P["x"]) for _ in range(3)]
    eps2, rc2 = prm["eps"] ** 2, prm["r_coll"] ** 2
    for i, j in _pairs(T, "pp"):
        d = [x[j] - x[i] for x in X]
        r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
        f = P["m"][j] * torch.clamp(r2, min=rc2).add_(eps2).pow_(-1.5)
        f[r2 == 0] = 0.0
        if rc2 > 0:
            t = torch.nonzero((r2 <= rc2) & (r2 > 0)).squeeze(1)
            it, jt, r = i[t], j[t], r2[t].sqrt()
            rv = sum(d[a][t] * (P["v" + s][jt] - P["v" + s][it]) for a, s in enumerate("xyz"))
            f[t] = f[t] * prm["G"] + P["m"][jt] / (P["m"][it] + P["m"][jt]) * (
                prm["kappa"] * (r - prm["r_coll"]) / r + prm["eta"] * rv / r2[t])
        for a in range(3):
            acc[a].index_add_(0, i, f * d[a])
    for i, c in _pairs(T, "pc"):
        d = [cen[a][c] - X[a][i] for a in range(3)]
        ri2 = 1.0 / (d[0] * d[0] + d[1] * d[1] + d[2] * d[2] + eps2)
        ri = ri2.sqrt()
        f, ri5 = M[c] * ri * ri2, ri * ri2 * ri2
        if prm["order"] == 2:
            q = [Q[k][c] for k in range(6)]
            u = [q[0] * d[0] + q[3] * d[1] + q[4] * d[2], q[3] * d[0] + q[1] * d[1] + q[5] * d[2],
                 q[4] * d[0] + q[5] * d[1] + q[2] * d[2]]
            f = f + 2.5 * (u[0] * d[0] + u[1] * d[1] + u[2] * d[2]) * ri5 * ri2
        for a in range(3):
            acc[a].index_add_(0, i, f * d[a] - (ri5 * u[a] if prm["order"] == 2 else 0.0))
    if central:
        f = prm["M_central"] * (X[0] ** 2 + X[1] ** 2 + X[2] ** 2) ** -1.5
        acc = [a - f * x for a, x in zip(acc, X)]
    return dict(zip(("ax", "ay", "az"), acc))


def _potential(T):
    P, prm = T["P"], T["prm"]
    M, cen, Q = _moments(T)
    X = [P["x"], P["y"], P["z"]]
    phi = torch.zeros_like(P["x"])
    eps2, rc2 = prm["eps"] ** 2, prm["r_coll"] ** 2
    for i, j in _pairs(T, "pp"):
        r2 = sum((x[j] - x[i]) ** 2 for x in X)
        s2 = torch.clamp(r2, min=rc2) + eps2
        v = 1.0 / s2.sqrt() + torch.clamp(rc2 - r2, min=0.0) / (2.0 * s2 * s2.sqrt())
        v[r2 == 0] = 0.0
        phi.index_add_(0, i, -P["m"][j] * v)
    for i, c in _pairs(T, "pc"):
        d = [X[a][i] - cen[a][c] for a in range(3)]
        R2 = d[0] ** 2 + d[1] ** 2 + d[2] ** 2 + eps2
        v = M[c] / R2.sqrt()
        if prm["order"] == 2:
            q = [Q[k][c] for k in range(6)]
            v = v + 0.5 * (q[0] * d[0] ** 2 + q[1] * d[1] ** 2 + q[2] * d[2] ** 2 +
                           2 * (q[3] * d[0] * d[1] + q[4] * d[0] * d[2] + q[5] * d[1] * d[2])) * R2 ** -2.5
        phi.index_add_(0, i, -v)
    return phi


def _advance(P, prm, steps):
    """`steps` kick-drift-kick steps of one particle set after the initial
    evaluation; lists rebuilt every rebuild_every evaluations."""
    T = _build(P, prm)
    a = _accelerations(T, True)
    c, s = math.cos(prm["omega"] * prm["dt"]), math.sin(prm["omega"] * prm["dt"])
    for k in range(1, steps + 1):
        P = T["P"]
        for f in "xyz":
            P["v" + f] = P["v" + f] + 0.5 * prm["dt"] * a["a" + f]
            P[f] = P[f] + prm["dt"] * P["v" + f]
        if prm["omega"]:
            for u, v in (("x", "y"), ("vx", "vy")):
                P[u], P[v] = c * P[u] + s * P[v], c * P[v] - s * P[u]
        if k % prm["rebuild_every"] == 0:
            T = _build(P, prm)
        a = _accelerations(T, True)
        for f in "xyz":
            T["P"]["v" + f] = T["P"]["v" + f] + 0.5 * prm["dt"] * a["a" + f]
    return {**T["P"], **a}


def _exact(c, P):
    prm, off = _params(c), _offsets(c)
    out = []
    for a, b in zip(off[:-1], off[1:]):
        p = {f: v[a:b] for f, v in P.items()}
        if c["op"] in ("steps", "host_steps"):
            out.append(_advance(p, prm, STEPS))
        elif c["op"] == "energy":
            T = _build(p, prm)
            out.append({"phi": _potential(T), **T["P"]})
        else:
            T = _build(p, prm)
            out.append({**T["P"], **_accelerations(T, False)})
    out = {f: torch.cat([o[f] for o in out]) for f in out[0]}
    if c["op"] == "forces":
        return {f: out[f] for f in ("ax", "ay", "az")}
    if c["op"] != "energy":
        return {f: out[f] for f in ALL}
    m, X = out["m"], torch.stack([out["x"], out["y"], out["z"]])
    V = torch.stack([out["vx"], out["vy"], out["vz"]])
    return {"phi": out["phi"], "W": float(0.5 * (m * out["phi"]).sum()), "mass": float(m.sum()),
            "kinetic": float((0.5 * m * (V * V).sum(0)).sum()),
            "central": float(-(prm["M_central"] * m / (X * X).sum(0).sqrt()).sum()),
            "momentum": (m * V).sum(1).cpu().numpy(),
            "angular_momentum": (m * torch.linalg.cross(X, V, dim=0)).sum(1).cpu().numpy()}


def exact(case, seed):
    c = case
    if c["op"] == "sort":
        key, idx = torch.sort(prepare(c, seed)["src"], stable=True)
        return {"key": key, "idx": idx.to(torch.int32)}
    evals = STEPS + 1 if c["op"] in ("steps", "host_steps") else 1
    if evals * c["n"] * sum(_interactions(c)) > 3e10:
        return None  # over about 20 seconds
    return _exact(c, _particles(c, seed))
