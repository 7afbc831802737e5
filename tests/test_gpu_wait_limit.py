"""A wait between a step's blocks that runs out (here after one poll) is
reported, stops the context's later kernels, and the next list starts clean:
the run from it equals that of a context that never waited too long."""
import numpy as np
import pytest

from ccmc_inputs import workload

pytestmark = pytest.mark.gpu

TIMEOUT = 5


def _start():
    """A list of several blocks in the scan and in the merge, with its state."""
    import paper_1807_03749_gb300 as ccmc

    w = workload("ueg14_m66_ccsdt_rs0.5", rs=1.0, fnc=False, target_pop=3e5, d0_init=4.5e4, tau=0.01)
    ctx = ccmc.from_workload(w)
    for _ in range(40):
        ctx.step(10)
        if ctx.list_size() > 4096:
            break
    bits, _, pop = ctx.get_list()
    state = ctx.get_state()
    assert len(pop) > 4096
    ctx.close()
    return w, bits, pop, state


def _restore(ctx, bits, pop, state):
    ctx.set_state(*state)
    ctx.set_list(bits, pop)


def _same(a, b):
    assert a.records(20) == b.records(20)
    assert all(np.array_equal(x, y) for x, y in zip(a.get_list(), b.get_list()))


@pytest.mark.parametrize("use_graph", [True, False])
@pytest.mark.parametrize("sort_all", [False, True])
def test_context_stops_and_restarts(use_graph, sort_all):
    torch = pytest.importorskip("torch")
    import paper_1807_03749_gb300 as ccmc

    w, bits, pop, state = _start()
    stream = torch.cuda.Stream()
    ctx = ccmc.from_workload(w, stream=stream.cuda_stream, use_graph=use_graph, sort_all=sort_all)
    want = ccmc.from_workload(w, stream=stream.cuda_stream, sort_all=sort_all)
    for c in (ctx, want):
        _restore(c, bits, pop, state)
    want.step(20)
    ctx.wait_limit(1)
    with pytest.raises(ccmc.CCMCError) as e:
        ctx.step(20)
    assert e.value.status == TIMEOUT
    # the error stays, and nothing runs on the unfinished step
    ctx.wait_limit(0)
    for call in (lambda: ctx.step(10), ctx.sync, ctx.energy, ctx.get_list):
        with pytest.raises(ccmc.CCMCError) as e:
            call()
        assert e.value.status == TIMEOUT
    _restore(ctx, bits, pop, state)
    ctx.step(20)
    _same(ctx, want)


def test_list_before_any_status_call():
    """The error word is overwritten unread: the barriers start clean all the same."""
    torch = pytest.importorskip("torch")
    import paper_1807_03749_gb300 as ccmc

    w, bits, pop, state = _start()
    stream = torch.cuda.Stream()
    ctx, want = (ccmc.from_workload(w, stream=stream.cuda_stream) for _ in range(2))
    for c in (ctx, want):
        _restore(c, bits, pop, state)
    want.step(20)
    ctx.wait_limit(1)
    ctx.step(3)                  # no shift boundary: nothing is reported
    _restore(ctx, bits, pop, state)
    ctx.wait_limit(0)            # (the limit outlasts the list)
    ctx.step(20)
    _same(ctx, want)


def test_batch_member_stops_and_restarts():
    torch = pytest.importorskip("torch")
    import paper_1807_03749_gb300 as ccmc

    w, bits, pop, state = _start()
    stream = torch.cuda.Stream()

    def members():
        return [ccmc.from_workload(dict(w, replica=q), stream=stream.cuda_stream) for q in range(3)]

    plain, ctxs = members(), members()
    for c in plain + ctxs:
        _restore(c, bits, pop, state)
    batch = ccmc.Batch(ctxs, stream.cuda_stream)
    ctxs[0].wait_limit(1)
    ctxs[2].wait_limit(1)
    with pytest.raises(ccmc.CCMCError) as e:
        batch.step(30)
    assert e.value.status == TIMEOUT
    for c in ctxs:               # the second timed-out member was never asked
        c.wait_limit(0)
        _restore(c, bits, pop, state)
    batch.step(30)
    for a, b in zip(plain, ctxs):
        a.step(30)
        _same(a, b)
    batch.close()
