"""List-build kernels at the edges of their tiles and of the rules that choose
them, against the oracle or numpy.  Keys, order, tree and lists are integers:
no tolerance.  FP32 forces: the 1e-5 gate."""
import numpy as np
import pytest

import oracle as orc
from paper_1907_02289_gb300 import synth
from _common import accel_of, assert_force_close, gpu_build, orc_params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


# sort tiles: 1536 keys below 600,000 keys, 4608 from there on; a tile's
# look-back takes 8 earlier tiles at a time (all there are, of the ninth tile)
@pytest.mark.parametrize("n", [1, 31, 1535, 1536, 1537, 8 * 1536, 9 * 1536, 9 * 1536 + 1, 17 * 1536 + 1, 599999,
                               600000, 600001])
@pytest.mark.parametrize("kind", ["random", "two digits", "sorted"])
def test_sort_tiles(n, kind):
    import torch
    from paper_1907_02289_gb300 import bh
    rng = np.random.default_rng(n)
    k = rng.integers(0, 1 << 63, n, dtype=np.uint64)
    if kind == "two digits":  # long runs of equal keys: stability, full digit bins
        k &= np.uint64(0x0100000000000001)
    elif kind == "sorted":
        k = np.sort(k)
    d = torch.from_numpy(k.view(np.int64).copy()).cuda()
    i = torch.empty(n, dtype=torch.int32, device="cuda")
    bh.bh_sort_keys_static(d, i, torch.empty_like(d), torch.empty_like(i))
    ref = np.argsort(k, kind="stable")
    assert np.array_equal(i.cpu().numpy().view(np.uint32), ref.astype(np.uint32))
    assert np.array_equal(d.cpu().numpy().view(np.uint64), k[ref])


def check_build(P, prm, precision=0):
    ref = orc.rebuild(P, orc_params(prm))
    ctx, D = gpu_build(P, prm, precision=precision)
    assert np.array_equal(ctx.bh_get_keys(len(P["x"]))[1], ref.perm)
    t = ctx.bh_get_tree()
    for f in ("level", "begin", "end", "parent", "first_child", "nchild", "qlo", "qhi"):
        assert np.array_equal(t[f], getattr(ref, f) if f in ("qlo", "qhi") else ref.tree[f]), f
    assert np.array_equal(ctx.bh_get_groups(), ref.groups)
    L = ctx.bh_get_lists()
    for f in ("pp_off", "P", "pc_off", "C"):
        assert np.array_equal(L[f], ref.lists[f]), f
    return ctx, D, ref


# tree tiles of 1024 particles; the window of a splitting cell is n_leaf + 1
@pytest.mark.parametrize("n", [2, 1023, 1024, 1025, 2049])
@pytest.mark.parametrize("n_leaf,n_g", [(1, 1), (1, 40), (2, 3), (7, 64), (40, 40), (300, 1000)])
def test_octree(n, n_leaf, n_g):
    P = synth.uniform_cube(n, n)
    P["x"][: n // 3] = 0.25  # a dense plane and a few coincident particles
    for f in ("x", "y", "z"):
        P[f][: min(n, 5)] = 0.75
    prm = dict(synth.PRESETS["cube4k"]["params"], n_leaf=n_leaf, n_g=n_g, theta=0.7)
    check_build(P, prm)


def test_patches_of_a_few_particles():
    """Patches below, at and above one sort tile and one tree tile."""
    from paper_1907_02289_gb300 import bh
    sizes = [1, 2, 1024, 1025, 4608, 4609, 9300, 3]
    off = np.concatenate([[0], np.cumsum(sizes)])
    parts = [synth.ring(s, 50 + q, phi_max=0.02) for q, s in enumerate(sizes)]
    _, prm = synth.make("ring1m_fp64", 16)
    prm = dict(prm, n_g=32)
    ctx = bh.Context(offsets=off, **prm)
    D = bh.Particles({f: np.concatenate([p[f] for p in parts]) for f in parts[0]})
    ctx.bh_build_tree(D)
    ctx.bh_make_lists()
    perm = ctx.bh_get_keys(int(off[-1]))[1].astype(np.int64)
    g, t, L = ctx.bh_get_groups(), ctx.bh_get_tree(), ctx.bh_get_lists()
    at = 0
    for q, p in enumerate(parts):
        ref = orc.rebuild(p, orc_params(prm))
        assert np.array_equal(perm[off[q]:off[q + 1]] - off[q], ref.perm)
        ng = len(ref.groups)
        assert np.array_equal(t["begin"][g[at:at + ng]].astype(np.int64) - off[q], ref.tree["begin"][ref.groups])
        for o, f in (("pp_off", "P"), ("pc_off", "C")):
            e0, e1 = L[o][at], L[o][at + ng]
            assert np.array_equal(t["begin"][L[f][e0:e1]].astype(np.int64) - off[q], ref.tree["begin"][ref.lists[f]])
        at += ng
    assert at == len(g)


def test_walk_of_long_lists():
    """theta = 0: every leaf is on every list, more than the 2048 entries that a
    warp holds (walked by one lane), and twice, so that the second build's
    single walk writes into slots."""
    P = synth.uniform_cube(6000, 3)
    prm = dict(synth.PRESETS["cube4k"]["params"], theta=0.0, n_leaf=2, n_g=200)
    ctx, D, ref = check_build(P, prm)
    assert np.diff(ref.lists["pp_off"]).max() > 2048
    ctx.bh_build_tree(D)
    ctx.bh_make_lists()
    L = ctx.bh_get_lists()
    for f in ("pp_off", "P", "pc_off", "C"):
        assert np.array_equal(L[f], ref.lists[f]), f


# a leaf tile holds 128 leaves and 640 particles in shared memory: "full" leaves of
# 5 fill it, one of 6 is one particle too many
@pytest.mark.parametrize("n,n_leaf,n_g", [(5, 8, 64), (1000, 1, 16), (20000, 5, 64), (20000, 6, 64), (20000, 64, 128),
                                          ("full", 5, 64), ("full + 1", 6, 64)])
def test_leaf_moments(n, n_leaf, n_g):
    if isinstance(n, str):
        rng = np.random.default_rng(4)
        site = np.repeat(np.arange(256), 5)
        site = np.append(site, 100) if n_leaf == 6 else site
        P, n = synth.uniform_cube(len(site), 6), len(site)
        for f in "xyz":
            P[f] = rng.random(256)[site]
        prm = dict(synth.PRESETS["cube4k"]["params"], order=2, n_leaf=n_leaf, n_g=n_g)
        ref = orc.rebuild(P, orc_params(prm))
        leaf = ref.tree["nchild"] == 0
        cnt = (ref.tree["end"].astype(int) - ref.tree["begin"])[leaf][np.argsort(ref.tree["begin"][leaf])]
        tiles = [cnt[k:k + 128].sum() for k in range(0, len(cnt), 128)]
        assert sorted(tiles) == ([640, 640] if n_leaf == 5 else [640, 641])
    else:
        P = synth.ring(n, n, phi_max=0.2)
        _, prm = synth.make("ring1m_fp64", 16)
        prm = dict(prm, n_leaf=n_leaf, n_g=n_g)
    ctx, D, ref = check_build(P, prm, precision=1)
    assert_force_close(accel_of(D), orc.tree_forces(ref, orc_params(prm)), 1e-5)
    mo = ctx.bh_get_moments()
    # FP32 records of FP64 sums over at most n particles: mass to n roundings,
    # centres (hi + lo) to the FP32 rounding of an offset within the node
    assert np.abs(mo["M"] / ref.mom["M"] - 1).max() <= n * 2.0 ** -24
    ext = max(np.ptp(P[f]) for f in "xyz")
    for f in ("cx", "cy", "cz"):
        assert np.abs(mo[f] - ref.mom[f]).max() <= 32 * 2.0 ** -24 * ext


def test_walk_of_longer_lists():
    """Lists of 2,000 to 16,000 entries, on a tree with chains of opened nodes down
    to the last level: a warp's buffer takes them in many pieces, down to
    pieces of one entry.  Twice, and through the step graphs."""
    from paper_1907_02289_gb300 import bh
    P = synth.uniform_cube(24000, 8)
    rng = np.random.default_rng(2)
    for c in range(40):  # clumps, of two particles in a last-level cell to a few hundred in many levels
        i = slice(300 * c, 300 * c + 300)
        for f in ("x", "y", "z"):
            P[f][i] = P[f][300 * c] + 10.0 ** -(1 + c % 7) * rng.random(300) ** 4
    prm = dict(synth.PRESETS["cube4k"]["params"], n_leaf=2, n_g=200)
    for theta in (0.0, 0.02, 0.2):
        ctx, D, ref = check_build(P, dict(prm, theta=theta))
        longest = (np.diff(ref.lists["pp_off"]) + np.diff(ref.lists["pc_off"])).max()
        assert longest > (12000 if theta == 0.0 else 2048)
        ctx.bh_build_tree(D)
        ctx.bh_make_lists()
        L = ctx.bh_get_lists()
        for f in ("pp_off", "P", "pc_off", "C"):
            assert np.array_equal(L[f], ref.lists[f]), f
        ctx.close()
    got = []
    for graph in (0, 1):
        ctx = bh.Context(**dict(prm, theta=0.2, rebuild_every=2))
        ctx.bh_set_tuning(graph=graph)
        D = bh.Particles(P)
        ctx.bh_step(D, 4)
        ctx.bh_sync()
        got.append(ctx.bh_get_lists())
        assert ctx.bh_get_counters()["n_graph_builds"] == 2 * graph
        ctx.close()
    for f in got[0]:
        assert np.array_equal(got[0][f], got[1][f]), f


def test_walk_time_of_long_lists():
    """A list entry costs about as much in lists that outgrow a warp's buffer
    (5.7 times as much while such a group was walked by one lane)."""
    from paper_1907_02289_gb300 import bh
    per = []
    for theta in (0.7, 0.4):
        P = synth.uniform_cube(100003, 3)
        ctx = bh.Context(**dict(synth.PRESETS["cube4k"]["params"], theta=theta, n_g=64, precision=1))
        D = bh.Particles(P)
        ctx.bh_set_timing(True)
        ms = []
        for _ in range(6):
            ctx.bh_get_timing(reset=True)
            ctx.bh_build_tree(D)
            ctx.bh_make_lists()
            ctx.bh_sync()
            ms.append(ctx.bh_get_counters()["stage_ms"]["lists"])
        L = ctx.bh_get_lists()
        n = np.diff(L["pp_off"]) + np.diff(L["pc_off"])
        assert (n.max() < 2048) == (theta == 0.7) and (theta == 0.7 or n.mean() > 2048)
        per.append(min(ms) / n.sum())
        ctx.close()
    assert per[1] < 2.5 * per[0], per
