"""What a restore writes to the device is ordered with the context's own stream:
it neither waits for the legacy stream (a context's stream does not wait for
that one either) nor leaves a copy behind on it."""
import numpy as np
import pytest

from ccmc_inputs import workload

pytestmark = pytest.mark.gpu


def test_restore_does_not_use_the_legacy_stream():
    torch = pytest.importorskip("torch")
    import paper_1807_03749_gb300 as ccmc

    stream = torch.cuda.Stream()
    w = workload("ueg14_m38_ccsd")
    ctx, want = ccmc.from_workload(w, stream=stream.cuda_stream), ccmc.from_workload(w, stream=stream.cuda_stream)
    want.step(20)
    ctx.step(10)
    bits, _, pop = ctx.get_list()
    state = ctx.get_state()
    for restore in (lambda: ctx.set_state(*state), lambda: ctx.set_list(bits, pop), lambda: ctx.wait_limit(0)):
        torch.cuda.synchronize()
        torch.cuda._sleep(400_000_000)           # some 0.2 s on the legacy stream
        asleep = torch.cuda.Event()
        asleep.record()
        restore()
        assert not asleep.query()
    ctx.step(10)
    assert all(np.array_equal(x, y) for x, y in zip(ctx.get_list(), want.get_list()))
    assert ctx.get_state() == want.get_state() and ctx.energy() == want.energy()
