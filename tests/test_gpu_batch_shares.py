"""A batch shares the blocks of its list kernels out in proportion to each
replica's list and records.  Lists of very different lengths together: every
replica's lists and records are those it gets alone, and a long list is not
left to the few blocks that an equal share would give it."""
import functools

import numpy as np
import pytest

from ccmc_inputs import workload

pytestmark = pytest.mark.gpu

STEPS = 20


@functools.lru_cache(maxsize=None)
def _long_list(nso, lmax, pop):
    """(workload, list, state) of a list grown with the original sampler."""
    import paper_1807_03749_gb300 as ccmc

    w = workload("ueg14_m38_ccsd", nso=nso, lmax=lmax, target_pop=pop, d0_init=0.15 * pop, list_capacity=200_000,
                 spawn_capacity=2_000_000)
    ctx = ccmc.from_workload(w)
    for _ in range(40):
        ctx.step(10)
        if ctx.energy()["n_total"] >= pop:
            break
    bits, _, pops = ctx.get_list()
    state = ctx.get_state()
    ctx.close()
    return w, bits, pops, state


SMALL = workload("ueg14_m38_ccsd", target_pop=2e3, d0_init=200.0, list_capacity=4096, spawn_capacity=16384)


def _context(kind, seed, stream):
    import paper_1807_03749_gb300 as ccmc

    if kind == "small":
        return ccmc.from_workload(dict(SMALL, seed=seed), stream=stream.cuda_stream)
    w, bits, pops, state = _long_list(66, 3, 3e5) if kind == "long" else _long_list(54, 3, 3e4)
    ctx = ccmc.from_workload(dict(w, seed=seed, spawn_capacity=200_000), stream=stream.cuda_stream)
    ctx.set_state(*state)
    ctx.set_list(bits, pops)
    return ctx


def _result(ctx):
    return ctx.get_list(), ctx.records(STEPS)


@functools.lru_cache(maxsize=None)
def _alone(kind, seed):
    import torch

    ctx = _context(kind, seed, torch.cuda.Stream())
    ctx.step(STEPS)
    out = _result(ctx)
    ctx.close()
    return out


# long lists: 20,000 entries (40 blocks alone); middle: thousands; small: one block
@pytest.mark.parametrize("longs,middles,smalls", [(1, 0, 300), (2, 3, 40), (0, 1, 700), (8, 0, 0), (40, 10, 20), (2, 0, 0),
                                                  (0, 0, 2), (1, 330, 0)])
def test_uneven_replicas_equal_plain(longs, middles, smalls):
    torch = pytest.importorskip("torch")
    import paper_1807_03749_gb300 as ccmc

    stream = torch.cuda.Stream()
    members = [("long", s) for s in range(longs)] + [("middle", s) for s in range(middles)] + [("small", s) for s in range(smalls)]
    members = members[1::2] + members[::2]       # the kinds' runs interleaved
    ctxs = [_context(k, s, stream) for k, s in members]
    batch = ccmc.Batch(ctxs, stream.cuda_stream)
    batch.step(STEPS)
    for (kind, seed), ctx in zip(members, ctxs):
        if seed in (0, 1, 2, 39, 299, 329, 699):
            (lists, recs), (want, want_recs) = _result(ctx), _alone(kind, seed)
            assert all(np.array_equal(x, y) for x, y in zip(lists, want)), (kind, seed)
            assert recs == want_recs, (kind, seed)
        else:
            assert len(ctx.records(STEPS)) == STEPS
    batch.close()
    for c in ctxs:
        c.close()


def test_one_long_list_among_many_small_ones():
    """Time of the list phases: at most three times what the long list and the
    small ones take by themselves, one after the other (ten times with equal
    shares)."""
    torch = pytest.importorskip("torch")
    import paper_1807_03749_gb300 as ccmc

    stream = torch.cuda.Stream()
    w, bits, pops, state = _long_list(114, 3, 1e6)

    def list_phases(long, smalls):
        ctxs = [ccmc.from_workload(w, stream=stream.cuda_stream) for _ in range(long)]
        for c in ctxs:
            c.set_state(*state)
            c.set_list(bits, pops)
        ctxs += [_context("small", s, stream) for s in range(smalls)]
        batch = ccmc.Batch(ctxs, stream.cuda_stream)
        batch.step(20)
        batch.profile(True)
        batch.step(20)
        ms, _, _ = batch.phase_times()
        batch.close()
        for c in ctxs:
            c.close()
        return sum(ms[p] for p in ("scan", "sort", "reduce", "merge"))

    assert len(pops) > 50_000
    apart = list_phases(1, 0) + list_phases(0, 200)
    together = list_phases(1, 200)
    assert together <= 3.0 * apart, (together, apart)
