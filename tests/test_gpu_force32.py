"""The FP32 force kernel's list loops at the sizes that pick their variants:
chunks of 1 to 3 slots with and without a tail, odd counts of list pairs,
cells flat along each axis (the kernel takes the quadrupole's xx entry out
of the matrix), with and without softening and contacts, and the work items:
windowed order, and chunk sizes, which change no bit.  Few items are cut to
chunks of 32, so chunks of 2 and 3 slots take sets of some 200,000 particles.
Tolerance: the FP32 gate, 1e-5 (rounding of ~30 units of 6e-8 per term, ~1e-6 of
a sum of ~1e3 terms; the quadrupole terms are 1e-3 to 1e-2 of the pull, so that
a wrong entry is 100 times the gate)."""
import numpy as np
import pytest

import oracle as orc
from paper_1907_02289_gb300 import synth
from _common import accel_of, assert_force_close, gpu_build, many_items, orc_params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


def check(P, prm):
    op = orc_params(prm)
    ctx, D = gpu_build(P, prm, precision=1)
    assert_force_close(accel_of(D), orc.tree_forces(orc.rebuild(P, op), op), 1e-5)
    ctx.close()


@pytest.mark.parametrize("n_g", [8, 31, 32, 33, 47, 48, 63, 64, 95, 97, 130])
def test_group_sizes_in_few_items(n_g):
    check(synth.uniform_cube(3001, n_g), dict(synth.PRESETS["cube4k"]["params"], order=2, n_g=n_g, theta=0.6))


MODES = {"plain": dict(eps=1e-3), "bare": dict(eps=0.0), "contacts": dict(eps=0.0, r_coll=2e-3),
         "soft contacts": dict(eps=1e-3, r_coll=2e-3)}


# groups of 38 to 73, 73 to 109 and 90 to 130 particles: chunks of one slot and a tail
# to three, and second chunks that are a tail
@pytest.mark.parametrize("n", [200001, 370003, 450007])
@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("mode", sorted(MODES))
def test_chunks_of_several_slots(n, order, mode):
    kappa, eta = synth.contact_params(1e-3)
    P = synth.uniform_cube(n, n)
    prm = dict(synth.PRESETS["cube4k"]["params"], order=order, n_g=140, theta=0.8, kappa=kappa, eta=eta, **MODES[mode])
    op = orc_params(prm)
    ref = orc.rebuild(P, op)
    aref = orc.tree_forces(ref, op)
    ctx, D = gpu_build(P, prm, precision=1, forces=False)
    for chunk in (96, 64):
        assert many_items(len(ref.groups), n, chunk)
        ctx.bh_set_tuning(chunk=chunk)
        ctx.bh_compute_forces(D, 1)
        assert_force_close(accel_of(D), aref, 1e-5)
        assert ("contacts" in mode) == (ctx.bh_get_counters()["n_contacts"] > 1000)
    ctx.close()


@pytest.mark.parametrize("axis", ["x", "y", "z"])
@pytest.mark.parametrize("eps", [0.0, 0.05])
def test_flat_cells(axis, eps):
    P = synth.uniform_cube(4000, 11)
    P[axis] = 0.5 + 0.02 * (P[axis] - 0.5)
    check(P, dict(synth.PRESETS["cube4k"]["params"], order=2, eps=eps, n_g=48, theta=0.8))


@pytest.mark.parametrize("chunk", [32, 96])
@pytest.mark.parametrize("window", [1, 63, 65, 91, 10000])
def test_windowed_items(window, chunk):
    """Groups of one to four chunks; the order of the items changes no bit."""
    P, prm = synth.uniform_cube(370003, 5), dict(synth.PRESETS["cube4k"]["params"], order=2, n_g=130)
    a = []
    for w in (0, window):
        ctx, D = gpu_build(P, prm, precision=1, forces=False)
        ctx.bh_set_tuning(chunk=chunk, order_window=w)
        ctx.bh_make_lists()
        ctx.bh_compute_forces(D, 1)
        a.append(accel_of(D))
        assert many_items(ctx.bh_get_sizes()["n_groups"], 370003, chunk)
        ctx.close()
    assert np.array_equal(a[0], a[1])


@pytest.mark.parametrize("shape", ["ring", "cube"])
def test_chunks_same_bits(shape):
    """Groups of one to three slots, with contacts and without."""
    if shape == "ring":
        P, prm = synth.ring(400000, 3, phi_max=0.05), dict(synth.PRESETS["ring16m_fp32"]["params"], n_g=100)
    else:
        P, prm = synth.uniform_cube(400000, 3), dict(synth.PRESETS["cube4k"]["params"], order=2, n_g=100)
    a = []
    for chunk in (96, 64, 32):
        ctx, D = gpu_build(P, prm, precision=1, forces=False)
        ctx.bh_set_tuning(chunk=chunk)
        ctx.bh_make_lists()
        ctx.bh_compute_forces(D, 1)
        a.append(accel_of(D))
        assert many_items(ctx.bh_get_sizes()["n_groups"], 400000, chunk)
        ctx.close()
    assert np.array_equal(a[0], a[1]) and np.array_equal(a[0], a[2])


def test_few_large_groups_keep_their_chunks():
    """3064 groups of 680 particles are 25,000 items of 96: cut to 32 (as few
    groups used to be) their lists would be staged three times as often."""
    P, prm = synth.ring(1 << 21, 3), dict(synth.PRESETS["ring16m_fp32"]["params"], n_g=2048)
    ctx, D = gpu_build(P, prm, precision=1)
    ms = {96: [], 32: []}
    for _ in range(3):
        for chunk in ms:
            ctx.bh_set_tuning(chunk=chunk)
            ctx.bh_set_timing(True)
            ctx.bh_get_timing(reset=True)
            for _ in range(3):
                ctx.bh_compute_forces(D, 1)
            ctx.bh_sync()
            t, k = ctx.bh_get_timing(reset=True)
            ms[chunk].append(t / k)
    assert min(ms[96]) < 0.92 * min(ms[32]), ms  # (3.6 and 4.3 ms)
    ctx.close()
