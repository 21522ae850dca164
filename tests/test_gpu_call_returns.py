"""What a call has done by the time it returns.  Work of the test's own, of a
tenth of a second, is put on the context's stream, so that a call that waits for the
stream, or returns before work that it should have waited for, is seen."""
import pytest

from paper_1907_02289_gb300 import synth

pytestmark = pytest.mark.gpu
SLEEP = 200_000_000  # GPU clock cycles, about 0.1 s


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


def context(P, precision=1, stream=None, **kw):
    from paper_1907_02289_gb300 import bh
    _, prm = synth.make("ring1m_fp64", 16)
    ctx = bh.Context(stream=stream, **dict(prm, precision=precision, **kw))
    return ctx, bh.Particles(P)


@pytest.mark.parametrize("precision", [0, 1])
def test_counters_do_not_wait_after_a_list_build(precision):
    import torch
    P = synth.ring(20000, 5, phi_max=0.2)
    s = torch.cuda.Stream()
    ctx, D = context(P, precision, s.cuda_stream, n_g=64)
    torch.cuda.synchronize()
    ctx.bh_build_tree(D)
    ctx.bh_make_lists()
    with torch.cuda.stream(s):
        torch.cuda._sleep(SLEEP)
    far = ctx.bh_get_counters()["n_pp_far"]
    assert not s.query(), "the counters waited for the stream"
    s.synchronize()
    assert far > 0 if precision else far == 0
    ctx.close()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("order", [1, 2])
def test_build_tree_hands_the_arrays_back(precision, order):
    """The particles may be written from another stream once bh_build_tree has
    returned: nothing of it still reads them (its moments did)."""
    import torch
    P = synth.ring(1 << 21, 7)
    ctx, D = context(P, precision, torch.cuda.Stream().cuda_stream, order=order)
    other = torch.cuda.Stream()
    got = []
    for spoil in (False, True):
        ctx.bh_build_tree(D)
        if spoil:
            with torch.cuda.stream(other):
                D.t["x"].add_(1.0)
        got.append({f: v.copy() for f, v in ctx.bh_get_moments().items()})
        torch.cuda.synchronize()
    for f, v in got[0].items():
        assert (v == got[1][f]).all(), f
    ctx.close()


@pytest.mark.parametrize("contacts", [False, True])
def test_first_forces_allocate_nothing(contacts):
    """The first evaluation finds its buffers: they are made with the lists."""
    import torch
    from paper_1907_02289_gb300 import bh
    kw = {} if contacts else {"r_coll": 0.0}
    small, D = context(synth.ring(1000, 9), **kw)  # (loads the kernels)
    small.bh_step(D, 0)
    small.bh_sync()
    ctx, D = context(synth.ring(1 << 20, 9), **kw)
    ctx.bh_build_tree(D)
    ctx.bh_make_lists()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    ctx.bh_compute_forces(D, bh.BH_FORCE_TREE_ONLY)
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == free
    ctx.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_a_new_stream_waits_for_the_lists(precision):
    """bh_make_lists may return while its lists are written; calls on a stream set
    then come after that."""
    import ctypes

    import torch
    ctx, D = context(synth.ring(1 << 22, 11), precision, (s := torch.cuda.Stream()).cuda_stream, n_g=64)
    ctx.bh_build_tree(D)
    ctx.bh_make_lists()
    torch.cuda.synchronize()
    ctx.bh_make_lists()
    new = torch.cuda.Stream()
    assert ctx.lib.bh_set_stream(ctx.h, ctypes.c_void_p(new.cuda_stream)) == 0
    ctx.bh_sync()
    assert s.query(), "the list build was still running"
    ctx.bh_compute_forces(D)
    ctx.bh_sync()
    assert new.query()
    ctx.close()
