"""Calls that read nothing back can be captured by the caller into a CUDA graph
of its own: evaluations without contacts, list-reusing steps, the static sort.
Replayed, they give the bits of the calls themselves."""
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


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("n", [20000, 300000])
def test_captured_evaluation_and_steps(precision, order, n):
    import torch
    from paper_1907_02289_gb300 import bh
    prm = dict(synth.PRESETS["ring16m_fp32"]["params"], n_g=64, precision=precision, order=order, r_coll=0.0,
               rebuild_every=1000)
    got = []
    for captured in (False, True):
        s = torch.cuda.Stream()
        ctx = bh.Context(stream=s.cuda_stream, **prm)
        D = bh.Particles(synth.ring(n, 12))
        torch.cuda.synchronize()
        ctx.bh_step(D, 1)
        ctx.bh_compute_forces(D)
        ctx.bh_sync()

        def work():
            ctx.bh_step(D, 2)
            ctx.bh_compute_forces(D, 1)

        if captured:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                work()
            for _ in range(3):
                g.replay()
        else:
            for _ in range(3):
                work()
        torch.cuda.synchronize()
        got.append(D.numpy())
        ctx.close()
    for f in got[0]:
        assert np.array_equal(got[0][f], got[1][f]), f


@pytest.mark.parametrize("n", [5000, 700000])
def test_captured_sort(n):
    import torch
    from paper_1907_02289_gb300 import bh
    rng = np.random.default_rng(n)
    src = torch.from_numpy(rng.integers(0, 1 << 62, n)).cuda()
    k, i = src.clone(), torch.empty(n, dtype=torch.int32, device="cuda")
    tmp = torch.empty_like(k), torch.empty_like(i)
    bh.bh_sort_keys_static(k, i, *tmp)  # (set-up)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        k.copy_(src)
        bh.bh_sort_keys_static(k, i, *tmp)
    for _ in range(2):
        g.replay()
    torch.cuda.synchronize()
    ref = torch.sort(src, stable=True)
    assert torch.equal(k, ref.values) and torch.equal(i.long(), ref.indices)
