"""The device memory of a small context follows its capacities: what does not is
the ring of 16,384 records."""
import pytest

from ccmc_inputs import workload

pytestmark = pytest.mark.gpu


def test_small_context():
    torch = pytest.importorskip("torch")
    import paper_1807_03749_gb300 as ccmc

    before = torch.cuda.memory_allocated()
    ctx = ccmc.from_workload(workload("ueg14_m38_ccsd"), target_pop=2e3, list_capacity=1024, spawn_capacity=4096,
                             use_torch_allocator=True)
    used = torch.cuda.memory_allocated() - before
    ctx.close()
    # some 200 bytes a list entry and 50 a spawned record, 100 KB of block
    # partials and orbital tables
    assert 16384 * 112 < used < 16384 * 112 + 1024 * 200 + 4096 * 50 + 200_000
    assert torch.cuda.memory_allocated() == before


@pytest.mark.parametrize("spawn_capacity", [4096, 4097, 70_000])
def test_records_up_to_the_spawn_capacity(spawn_capacity):
    """As many sorting blocks as the buffer's records can have: the sort of a
    buffer that is nearly full gives the list of a larger one."""
    import numpy as np

    import paper_1807_03749_gb300 as ccmc

    w = workload("ueg14_m38_ccsd", target_pop=50.0 * spawn_capacity, d0_init=2.0 * spawn_capacity, sort_all=True)
    big = ccmc.from_workload(w, spawn_capacity=1_000_000)
    steps = 0
    while steps < 200:
        big.step(1)
        steps += 1
        if big.records(1)[-1]["n_spawned"] > spawn_capacity:
            break
    steps -= 1                                # the last step whose records fit
    assert steps > 0
    ctx, want = (ccmc.from_workload(w, spawn_capacity=c) for c in (spawn_capacity, 1_000_000))
    for c in (ctx, want):
        c.step(steps)
    assert all(np.array_equal(x, y) for x, y in zip(ctx.get_list(), want.get_list()))
    rec = ctx.records(1)[-1]
    assert rec == want.records(1)[-1] and rec["n_spawned"] > spawn_capacity // 4
