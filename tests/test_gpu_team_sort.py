"""The annihilation's sort and reduction at the edges of its forms: ranked by
counting (up to 256 records), one block's tile (up to 4,096), several blocks;
one to eight digits, remainders of the 512 threads, runs of equal keys across
warps, tiles and blocks.  Equal to numpy's stable sort and integer sums."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 31, 33, 255, 256, 257, 511, 513, 1025, 4095, 4096, 4097, 5121, 12289, 65535, 65536])
@pytest.mark.parametrize("bits,distinct", [(1, 2), (9, 300), (10, 1 << 10), (27, 1 << 20), (33, 1), (64, 1 << 40)])
def test_sort_and_reduce_edges(n, bits, distinct):
    import torch

    import paper_1807_03749_gb300 as ccmc

    lib = ccmc.load()
    rng = np.random.default_rng(1000 * n + bits)
    top = (1 << bits) - 1
    keys = rng.integers(0, min(distinct, top + 1), size=n, dtype=np.uint64) * np.uint64(max(1, top // max(1, distinct)))
    keys[rng.integers(0, n)] = np.uint64(top)     # the largest key of the range
    pops = rng.integers(-(1 << 40), 1 << 40, size=n, dtype=np.int64)
    want, inv = np.unique(keys, return_inverse=True)
    sums = np.zeros(len(want), dtype=np.int64)
    np.add.at(sums, inv, pops)
    dk, dp = torch.from_numpy(keys.view(np.int64)).cuda(), torch.from_numpy(pops).cuda()
    for _ in range(2):                            # the barriers are left as found
        ok, op = torch.full_like(dk, -1), torch.full_like(dp, 77)
        m = ctypes.c_size_t(0)
        torch.cuda.synchronize()
        assert lib.ccmc_reduce_records_noalloc(dk.data_ptr(), dp.data_ptr(), n, bits, ok.data_ptr(), op.data_ptr(),
                                               ctypes.byref(m), None) == 0
        assert m.value == len(want)
        assert np.array_equal(ok[: m.value].cpu().numpy().view(np.uint64), want)
        assert np.array_equal(op[: m.value].cpu().numpy(), sums)
    assert np.array_equal(dk.cpu().numpy().view(np.uint64), keys)   # inputs are read only


def _lists(w, nsteps, **over):
    import paper_1807_03749_gb300 as ccmc

    ctx = ccmc.from_workload(dict(w, **over))
    ctx.step(nsteps)
    return ctx.get_list(), ctx.records()


@pytest.mark.parametrize("sort_all", [False, True])
def test_team_sizes_give_one_result(sort_all):
    """A batch shares the GPU between its replicas' teams (down to one block
    each), a context alone uses all blocks, and six-bit digits take more
    passes: the same lists and records."""
    import torch

    import paper_1807_03749_gb300 as ccmc
    from ccmc_inputs import workload

    w = workload("ueg14_m66_ccsdt_rs5", target_pop=1e5, d0_init=2e4, tau=0.01, multispawn=True, sort_all=sort_all)
    (b0, k0, p0), r0 = _lists(w, 30)
    (b1, k1, p1), r1 = _lists(w, 30, radix_bits=6)
    assert np.array_equal(b0, b1) and np.array_equal(p0, p1) and r0 == r1
    stream = torch.cuda.Stream()
    small = workload("ueg14_m38_ccsd", target_pop=2e3, d0_init=200.0)
    ctxs = [ccmc.from_workload(w, stream=stream.cuda_stream)]
    ctxs += [ccmc.from_workload(dict(small, seed=s), stream=stream.cuda_stream) for s in range(320)]
    batch = ccmc.Batch(ctxs, stream.cuda_stream)
    batch.step(30)
    bits, keys, pop = ctxs[0].get_list()
    assert np.array_equal(keys, k0) and np.array_equal(pop, p0) and ctxs[0].records() == r0
