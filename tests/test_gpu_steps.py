"""Several steps in one call take the closing kick of a step and the next
kick-drift in one pass: the same bits as the steps one call each (every
operation keeps its own rounding), eager and mixed with graph steps."""
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


@pytest.mark.parametrize("n", [1, 255, 257, 5000])
@pytest.mark.parametrize("omega,graph", [(0.0, 0), (1.0, 0), (0.0, 2)])
def test_steps_in_one_call(n, omega, graph):
    from paper_1907_02289_gb300 import bh
    P = synth.ring(n, 17, phi_max=1e-3)
    prm = dict(synth.PRESETS["ring16m_fp32"]["params"], n_g=64, omega=omega)
    got = []
    for calls in ((6,), (1,) * 6):
        ctx = bh.Context(**prm)
        ctx.bh_set_tuning(graph=graph)
        D = bh.Particles(P)
        for k in calls:
            ctx.bh_step(D, k)
        ctx.bh_sync()
        got.append(D.numpy())
        ctx.close()
    for f in ("x", "y", "z", "vx", "vy", "vz", "ax", "ay", "az"):
        assert np.array_equal(got[0][f], got[1][f]), f
