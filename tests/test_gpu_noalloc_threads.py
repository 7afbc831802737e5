"""Calls of ccmc_reduce_records_noalloc from several threads on one stream: the
GPU runs them one after another while their host parts overlap.  Every call
gets its own count."""
import ctypes
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [(1, 200), (300, 4096), (5000, 70), (12000, 65536)])
def test_threads_on_one_stream_get_their_own_counts(sizes):
    torch = pytest.importorskip("torch")
    import paper_1807_03749_gb300 as ccmc

    lib = ccmc.load()
    stream = torch.cuda.Stream()
    wrong = []

    def work(n, threads_id):
        torch.cuda.set_device(0)
        rng = np.random.default_rng(100 * n + threads_id)
        keys = rng.integers(0, max(2, n // 3), size=n, dtype=np.uint64)
        pops = rng.integers(-1000, 1000, size=n, dtype=np.int64)
        want, inv = np.unique(keys, return_inverse=True)
        sums = np.zeros(len(want), dtype=np.int64)
        np.add.at(sums, inv, pops)
        dk, dp = torch.from_numpy(keys.view(np.int64)).cuda(), torch.from_numpy(pops).cuda()
        ok, op = torch.empty_like(dk), torch.empty_like(dp)
        m = ctypes.c_size_t(0)
        torch.cuda.synchronize()
        gate.wait()
        for _ in range(400):
            st = lib.ccmc_reduce_records_noalloc(dk.data_ptr(), dp.data_ptr(), n, 20, ok.data_ptr(), op.data_ptr(),
                                                 ctypes.byref(m), stream.cuda_stream)
            if st != 0 or m.value != len(want):
                wrong.append((n, st, m.value, len(want)))
                return
        if not (np.array_equal(ok[: m.value].cpu().numpy().view(np.uint64), want)
                and np.array_equal(op[: m.value].cpu().numpy(), sums)):
            wrong.append((n, "values"))

    threads = [threading.Thread(target=work, args=(n, q)) for q, n in enumerate(sizes + sizes)]
    gate = threading.Barrier(len(threads))
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong
