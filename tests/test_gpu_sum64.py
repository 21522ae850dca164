"""FP64 force and potential kernels at the edges of their work split: groups
are cut along the binary digits of their size, the largest item grows with
the particle count (1 to 8 particles), and each item's lists are split over
the remaining lanes; separations outside the range of the inverse-square-root
series take the library functions.  Tolerance: the FP64 gate, 1e-12 of every
value (a sum of ~1e3 terms of either sign in another order: ~1e-14)."""
import numpy as np
import pytest

import oracle as orc
from paper_1907_02289_gb300 import bh, synth
from _common import accel_of, assert_force_close, gpu_build, orc_params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


def check(P, prm, tol=1e-12):
    import torch
    op = orc_params(prm)
    ref = orc.rebuild(P, op)
    ctx, D = gpu_build(P, prm, precision=0)
    aref = orc.tree_forces(ref, op)
    unit = np.abs(aref).max()  # (the squares of 1e180 would not fit the metric's norms)
    if unit == 0.0:  # a particle alone
        assert not accel_of(D).any()
    else:
        assert_force_close(accel_of(D) / unit, aref / unit, tol)
    phi = torch.empty(len(P["x"]), dtype=torch.float64, device="cuda")
    W = ctx.bh_compute_potential(D, phi)
    pref = orc.tree_potential(ref, op)
    if len(pref) == 1:
        assert W == 0.0 and float(phi[0]) == 0.0 and pref[0] == 0.0
        return
    assert np.abs(phi.cpu().numpy() / pref - 1.0).max() <= tol
    assert abs(W / (0.5 * (ref.P["m"] * pref).sum()) - 1.0) <= tol
    ctx.close()


# the largest item grows at 20,000, 40,000 and 80,000 particles
@pytest.mark.parametrize("n", [1, 33, 4097, 19999, 20001, 39999, 40001, 79999, 80001])
@pytest.mark.parametrize("order,eps", [(1, 1e-3), (2, 0.0)])
def test_item_sizes(n, order, eps):
    prm = dict(synth.PRESETS["cube4k"]["params"], order=order, eps=eps, theta=0.7, n_g=40)
    check(synth.uniform_cube(n, n), prm)


@pytest.mark.parametrize("n_g", [8, 31, 33, 100])
def test_group_sizes_with_contacts(n_g):
    _, prm = synth.make("ring1m_fp64", 16)
    P = synth.ring(6000, 9, r_in=0.99995, r_out=1.00005, phi_max=4e-4, sigma_z=5e-6)
    check(P, dict(prm, n_g=n_g, theta=0.6))


def test_group_above_n_g():
    """Coincident particles: one leaf far above n_g, in whole items and a remainder."""
    P = synth.uniform_cube(500, 4)
    for f in ("x", "y", "z"):
        P[f][:333] = 0.5
    check(P, dict(synth.PRESETS["cube4k"]["params"], n_g=16))


@pytest.mark.parametrize("scale", [1e-100, 1e-91, 1e-60, 1e60, 1e90, 1e100])
def test_separation_range(scale):
    """r^2 from 1e-204 to 1e200: both sides of the series' range (2^-600 to 2^600)."""
    P = synth.uniform_cube(700, 5)
    for f in ("x", "y", "z"):
        P[f] = P[f] * scale
    check(P, dict(synth.PRESETS["cube4k"]["params"], eps=0.0, order=1))
