"""The batch tuner times only candidates that differ: the blocks of the attempt
and owner-table kernels are tried only if a member uses these kernels."""
import pytest

from ccmc_inputs import workload

pytestmark = pytest.mark.gpu

WORK, TILE, DIGIT = 4, 5, 2   # candidates of the stages


@pytest.mark.parametrize("member,steps", [
    (dict(), TILE + DIGIT),
    (dict(fnc=True), WORK + TILE + DIGIT),
    (dict(fnc=True, multispawn=True), WORK + TILE + DIGIT),
    (dict(n_ranks=4, nu_move=3), WORK + TILE + DIGIT),
])
def test_tuning_steps(member, steps):
    torch = pytest.importorskip("torch")
    import paper_1807_03749_gb300 as ccmc

    stream = torch.cuda.Stream()
    w = workload("ueg14_m38_ccsd")
    ctxs = [ccmc.from_workload(w, replica=0), ccmc.from_workload(dict(w, **member), replica=1)]
    batch = ccmc.Batch(ctxs, stream.cuda_stream)
    batch.step(steps - 1)
    assert batch.info()["tunings"] == 0
    batch.step(1)
    assert batch.info()["tunings"] == 1
    batch.close()
