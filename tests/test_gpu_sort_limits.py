"""The bounds of the key sort's look-back: 64-bit counts (in use from 2^27
particles) give the order of 32-bit ones, and a wait that runs out is reported, with
the particles left alone.  Keys and orders are integers: no tolerance."""
import numpy as np
import pytest

from paper_1907_02289_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


def _prm(**kw):
    return dict(synth.PRESETS["ring16m_fp32"]["params"], n_g=64, **kw)


@pytest.mark.parametrize("sizes", [[1], [4608], [4609], [65537], [600001], [2, 4608, 4609, 1, 50000, 9300]])
def test_wide_counts_give_the_same_order(sizes):
    from paper_1907_02289_gb300 import bh
    n, off = sum(sizes), np.concatenate([[0], np.cumsum(sizes)])
    P = synth.ring(n, 3)
    got = []
    for wide in (1 << 27, 1):
        ctx = bh.Context(offsets=off if len(sizes) > 1 else None, **_prm())
        ctx.bh_set_sort_limits(wide_from=wide)
        ctx.bh_build_tree(bh.Particles(P))
        got.append(ctx.bh_get_keys(n))
        ctx.close()
    for a, b in zip(*got):
        assert np.array_equal(a, b)


def test_limits_changed_between_graph_steps():
    """The captured step is made again, with the scratch of the wider counts."""
    from paper_1907_02289_gb300 import bh
    P, got = synth.ring(700000, 6), []
    for wide in (False, True):
        ctx = bh.Context(**_prm())
        ctx.bh_set_tuning(graph=1)
        D = bh.Particles(P)
        ctx.bh_step(D, 6)
        if wide:
            ctx.bh_set_sort_limits(wide_from=1)
        ctx.bh_step(D, 6)
        ctx.bh_sync()
        assert ctx.bh_get_counters()["n_graph_builds"] == 3
        got.append(D.numpy())
        ctx.close()
    for f in got[0]:
        assert np.array_equal(got[0][f], got[1][f]), f


def test_a_wait_that_runs_out_is_reported():
    """No poll allowed: every tile but the first gives up."""
    from paper_1907_02289_gb300 import bh
    P = synth.ring(600001, 4)
    ctx = bh.Context(**_prm())
    D = bh.Particles(P)
    ctx.bh_set_sort_limits(polls=0)
    with pytest.raises(bh.BHError) as e:
        ctx.bh_build_tree(D)
    assert e.value.code == bh.BH_E_TIMEOUT
    out = D.numpy()
    for f in ("x", "y", "z", "vx", "vy", "vz", "m", "id"):
        assert np.array_equal(out[f], P[f]), f
    with pytest.raises(bh.BHError):
        ctx.bh_make_lists()
    ctx.bh_set_sort_limits()
    ctx.bh_build_tree(D)
    keys, perm = ctx.bh_get_keys(600001)
    assert (np.diff(keys.astype(np.int64)) >= 0).all() and np.array_equal(np.sort(perm), np.arange(600001))
    ctx.close()


def test_a_wait_that_runs_out_in_a_graph_step():
    """The step ends after its kick and drift; nothing is built on unsorted keys."""
    from paper_1907_02289_gb300 import bh
    P = synth.ring(600001, 5)
    ctx = bh.Context(**_prm())
    ctx.bh_set_tuning(graph=1)
    D = bh.Particles(P)
    ctx.bh_step(D, 4)  # evaluations 0..4: a list-constructing graph step at 4
    assert ctx.bh_get_counters()["n_graph_builds"] == 1
    ctx.bh_step(D, 3)
    ctx.bh_sync()
    before = D.numpy()
    ctx.bh_set_sort_limits(polls=0)
    with pytest.raises(bh.BHError) as e:
        ctx.bh_step(D, 1)
    assert e.value.code == bh.BH_E_TIMEOUT
    after = D.numpy()
    assert np.array_equal(before["id"], after["id"]) and np.array_equal(before["m"], after["m"])
    dt = ctx.params.dt
    for f in "xyz":
        v = before["v" + f] + 0.5 * dt * before["a" + f]
        assert np.allclose(after["v" + f], v, rtol=0, atol=1e-15)  # (|v| <= 1, a few roundings)
        assert np.allclose(after[f], before[f] + dt * v, rtol=0, atol=1e-15)
    with pytest.raises(bh.BHError) as e:
        ctx.bh_compute_forces(D)
    assert e.value.code == bh.BH_E_STATE
    ctx.bh_set_sort_limits()
    ctx.bh_step(D, 8)
    ctx.bh_sync()
    assert np.array_equal(np.sort(D.numpy()["id"]), np.sort(P["id"]))
    ctx.close()


def test_static_sort_reports_a_wait_that_ran_out():
    import torch
    from paper_1907_02289_gb300 import bh
    k = np.random.default_rng(1).integers(0, 1 << 63, 600001, dtype=np.uint64)
    d = torch.from_numpy(k.view(np.int64).copy()).cuda()
    i = torch.empty(len(k), dtype=torch.int32, device="cuda")
    tmp = torch.empty_like(d), torch.empty_like(i)
    assert bh.bh_sort_static_status() == bh.BH_OK
    bh.bh_sort_keys_static_bounded(d.clone(), i, *tmp, polls=0)
    with pytest.raises(bh.BHError) as e:
        bh.bh_sort_static_status()
    assert e.value.code == bh.BH_E_TIMEOUT
    assert bh.bh_sort_static_status() == bh.BH_OK  # (told once)
    for sort in (lambda: bh.bh_sort_keys_static(d, i, *tmp),
                 lambda: bh.bh_sort_keys_static_bounded(d, i, *tmp, polls=1 << 22)):
        d.copy_(torch.from_numpy(k.view(np.int64)))
        sort()
        assert bh.bh_sort_static_status() == bh.BH_OK
        ref = np.argsort(k, kind="stable")
        assert np.array_equal(i.cpu().numpy().view(np.uint32), ref.astype(np.uint32))
        assert np.array_equal(d.cpu().numpy().view(np.uint64), k[ref])


def test_limits_out_of_range_are_refused():
    import torch
    from paper_1907_02289_gb300 import bh
    ctx = bh.Context(**_prm())
    for kw in (dict(wide_from=0), dict(wide_from=(1 << 27) + 1), dict(polls=-1), dict(polls=(1 << 22) + 1)):
        with pytest.raises(bh.BHError) as e:
            ctx.bh_set_sort_limits(**kw)
        assert e.value.code == bh.BH_E_INVAL
    t = torch.zeros(8, dtype=torch.int64, device="cuda"), torch.zeros(8, dtype=torch.int32, device="cuda")
    with pytest.raises(bh.BHError) as e:
        bh.bh_sort_keys_static_bounded(t[0], t[1], t[0].clone(), t[1].clone(), polls=-1)
    assert e.value.code == bh.BH_E_INVAL
    ctx.close()
