"""Co-location calls of several threads with different numbers of processors
(different sizes of the pair kernel's shared memory)."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_threads_with_few_and_many_processors():
    torch = pytest.importorskip("torch")
    import paper_1807_03749_gb300 as ccmc

    rng = np.random.default_rng(11)
    words = rng.integers(0, 1 << 62, size=(40, 2), dtype=np.uint64)
    ranks = [1, 2, 65535, 40000]
    want = {r: ccmc.colocation(words, r, 3, [50, 300]) for r in ranks}
    failed = []

    def work(r):
        torch.cuda.set_device(0)
        stream = torch.cuda.Stream()
        gate.wait()
        try:
            for _ in range(1500):
                got = ccmc.colocation(words, r, 3, [50, 300], stream=stream.cuda_stream)
                assert all(np.array_equal(x, y) for x, y in zip(got, want[r]))
        except Exception as e:
            failed.append((r, repr(e)))

    threads = [threading.Thread(target=work, args=(r,)) for r in ranks]
    gate = threading.Barrier(len(threads))
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed
