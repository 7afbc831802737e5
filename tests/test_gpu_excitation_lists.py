"""Lockstep with the oracle where the excitation lists have their edges:
clusters of up to six excitors and six holes (l = 4), level 1 only, odd
electron numbers, spin-orbitals past 255, every sampler; a spawn cutoff that
is no power of two (rounding in FP64) and multi-spawn thresholds other than
one; four and five-word determinants."""
import numpy as np
import pytest

import oracle
from ccmc_inputs import molecule_integrals

pytestmark = pytest.mark.gpu

FIELDS = ["n0", "ntot", "n_sel", "n_visit", "n_attempts", "n_spawned", "ntot_after", "nocc_after", "n_keys"]
BASE = dict(tau=0.01, target_pop=2000.0, d0_init=300.0, shift_a=10, zeta=0.05, spawn_cutoff=2.0 ** -7, a_thresh=1.0,
            seed=11, replica=2, fnc=False, multispawn=False)


def _lockstep(kind, nel, nso, lmax, nsteps, precision="fp64", **over):
    import paper_1807_03749_gb300 as ccmc

    w = dict(BASE, **over)
    if kind == "ueg":
        so = oracle.System.ueg(nel, nso, 1.0, lmax)
        more = {"rs": 1.0}
    else:
        h1, eri = molecule_integrals(norb=nso // 2, nocc=(nel + 1) // 2, seed=5, scale=0.1)
        so = oracle.System.generic(nel, h1, eri, lmax)
        more = {"h1": h1, "eri": eri}
    if precision == "fp32":
        so.set_fp32()
    sim = oracle.Sim(so, **w)
    # room for the largest space, which keeps growing
    ctx = ccmc.Context(kind, nel, nso, lmax, precision=precision, list_capacity=1 << 20, spawn_capacity=1 << 22, **more, **w)
    for _ in range(nsteps):
        rec = sim.step().as_dict()
        ctx.step(1)
        got = ctx.records()[-1]
        assert all(rec[f] == got[f] for f in FIELDS), [(f, rec[f], got[f]) for f in FIELDS]
        assert abs(rec["e_num"] - got["e_num"]) <= 1e-12 * max(abs(rec["e_num"]), 1e-300)
    ob, ok, op = sim.get_list()
    gb, gk, gp = ctx.get_list()
    assert np.array_equal(ob, gb) and np.array_equal(ok, gk) and np.array_equal(op, gp)
    return len(gk)


@pytest.mark.parametrize("nel,nso,lmax", [(6, 16, 4), (5, 14, 3), (7, 18, 4), (6, 20, 1), (2, 12, 2)])
@pytest.mark.parametrize("fnc,ms", [(False, False), (True, False), (True, True)])
def test_generic_systems(nel, nso, lmax, fnc, ms):
    _lockstep("generic", nel, nso, lmax, 40, fnc=fnc, multispawn=ms)


@pytest.mark.parametrize("nso,lmax,words", [(38, 4, 1), (246, 2, 4), (294, 3, 5), (358, 4, 6)])
@pytest.mark.parametrize("fnc", [False, True])
def test_gas_systems(nso, lmax, words, fnc):
    n = _lockstep("ueg", 14, nso, lmax, 15, fnc=fnc, multispawn=fnc, d0_init=1000.0, target_pop=1e4)
    assert n > 50 and (nso + 63) // 64 == words


@pytest.mark.parametrize("cutoff", [0.01, 0.0])
@pytest.mark.parametrize("kind,nel,nso,lmax", [("generic", 6, 16, 3), ("ueg", 14, 38, 2)])
def test_spawn_cutoffs(kind, nel, nso, lmax, cutoff):
    _lockstep(kind, nel, nso, lmax, 40, spawn_cutoff=cutoff)


@pytest.mark.parametrize("a_thresh", [0.5, 2.75])
def test_multispawn_thresholds(a_thresh):
    _lockstep("generic", 6, 16, 3, 40, multispawn=True, a_thresh=a_thresh)
    _lockstep("ueg", 14, 38, 3, 25, multispawn=True, fnc=True, a_thresh=a_thresh, d0_init=1000.0)


def test_single_precision_generic_level_four():
    _lockstep("generic", 6, 16, 4, 40, precision="fp32")


@pytest.mark.parametrize("ranks,nu", [(3, 0), (7, 2)])
def test_simulated_processors_level_four(ranks, nu):
    _lockstep("generic", 6, 16, 4, 40, n_ranks=ranks, nu_move=nu)
