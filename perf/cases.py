"""Performance cases of the CCMC library: what a program asks of it.

A wavefunction is restored from host memory, advanced by one or more shift
periods and read back (list, estimators, per-step records) -- the life of a
run between two checkpoints -- for the electron gas and the molecule-like
Hamiltonian, with every sampler, both precisions, the simulated distribution
over processors and the batched form; beside it the library's two standalone
calls, the sort-and-reduce of spawned records and the co-location statistics.

The starting wavefunctions are grown by the library itself from the reference
(every trajectory is reproducible bit for bit) and then scaled to the case's
population: t_HF exp(T/t_HF) scales as a whole.
"""
import ctypes
import functools
import math

import numpy as np
import torch

import paper_1807_03749_gb300 as ccmc
from ccmc_inputs import batched_replicas, molecule_integrals

# occupied excitors of a saturated list, by (spin-orbitals, truncation level)
SATURATED = {(38, 2): 289, (54, 2): 537, (66, 2): 741, (114, 2): 1797, (162, 2): 15769, (186, 2): 3813,
             (38, 3): 2665, (54, 3): 12433, (66, 3): 22969, (114, 3): 108753}


def _gas(orbitals, level, sampler, population, steps, **more):
    case = {"kind": "steps", "system": "gas", "electrons": 14, "orbitals": orbitals, "level": level, "rs": 1.0,
            "sampler": sampler, "population": population, "tau": 0.01, "precision": "fp64",
            "processors": 1, "move": 0, "steps": steps}
    case.update(more)
    return case


def _molecule(level, sampler, population, steps, **more):
    case = {"kind": "steps", "system": "molecule", "electrons": 20, "orbitals": 82, "level": level, "rs": 0.0,
            "sampler": sampler, "population": population, "tau": 2.0e-6, "precision": "fp64",
            "processors": 1, "move": 0, "steps": steps}
    case.update(more)
    return case


def listed():
    return [
        # the smallest system a user starts with: launches and latency
        dict(_gas(38, 2, "original", 2.0e4, 50), name="gas38_ccsd"),
        # the paper's bias study: full non-composite sampling, 32 simulated processors
        dict(_gas(66, 3, "full", 2.0e5, 50, rs=5.0, tau=0.001, processors=32, move=5),
             name="gas66_ccsdt_full_32_processors"),
        # the recommended sampler at production size, two-word determinants
        dict(_gas(114, 3, "multispawn", 1.0e6, 20, tau=0.005), name="gas114_ccsdt_multispawn"),
        # the paper's published-energy system: six-word determinants, an unsaturated list
        dict(_gas(358, 4, "multispawn", 3.0e6, 5, tau=0.003), name="gas358_ccsdtq_multispawn"),
        # the single-precision form at scale: compute, a tiny list
        dict(_gas(162, 2, "original", 1.0e8, 5, electrons=54, precision="fp32"), name="gas162_ccsd_fp32"),
        # a mid-sized molecule run stepped one step at a time between reads
        dict(_molecule(3, "full", 3.0e5, 1), name="molecule82_ccsdt_full_one_step"),
        # the largest run: random gathers from a list far beyond the caches
        dict(_molecule(4, "original", 2.0e7, 10), name="molecule82_ccsdtq"),
        # a parameter scan: replicas of uneven size stepped together
        {"kind": "batch", "replicas": 64, "grow": 100, "steps": 10, "name": "batch64_gas"},
        # standalone sort-and-reduce: one buffer's worth, and a small odd one
        {"kind": "reduce", "records": 65536, "key_bits": 27, "per_key": 4.0, "name": "reduce_65536_records"},
        {"kind": "reduce", "records": 3001, "key_bits": 33, "per_key": 1.5, "name": "reduce_3001_records"},
        # co-location statistics of the paper's 3,813-excitor space
        {"kind": "colocation", "excitors": 3813, "orbitals": 186, "processors": 32, "move": 4, "iterations": 4096,
         "checkpoints": 8, "name": "colocation_3813"},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["gas", "gas", "gas", "molecule", "molecule", "fp32", "batch", "reduce", "colocation"])
    if kind == "gas":
        orbitals, level = rng.choice([(38, 2), (38, 3), (54, 3), (66, 2), (66, 3), (114, 2), (114, 3), (186, 2),
                                      (358, 4)])
        sampler = rng.choice(["original", "full", "multispawn"])
        rs = round(_log(rng, 0.5, 5.0) if sampler != "multispawn" else _log(rng, 0.5, 1.0), 3)
        processors = rng.choice([1, 1, 1, rng.randrange(2, 97)])
        # the largest space keeps growing at these populations: fewer steps
        steps = rng.choice([1, 3, 5] if orbitals == 358 else [1, 10, 20, 30])
        return _gas(orbitals, level, sampler, float(int(_log(rng, 1.0e4, 3.0e6))), steps, rs=rs,
                    tau=0.003 if orbitals >= 114 else 0.005, processors=processors,
                    move=rng.randrange(0, 7) if processors > 1 else 0)
    if kind == "fp32":
        electrons, orbitals, level = rng.choice([(14, 38, 3), (14, 66, 3), (14, 114, 2), (54, 162, 2)])
        return _gas(orbitals, level, "original", float(int(_log(rng, 1.0e5, 5.0e7))), 10, electrons=electrons,
                    precision="fp32")
    if kind == "molecule":
        return _molecule(rng.choice([2, 3, 4]), rng.choice(["original", "original", "full"]),
                         float(int(_log(rng, 3.0e4, 6.0e6))), rng.choice([1, 10]))
    if kind == "batch":
        return {"kind": "batch", "replicas": rng.randrange(3, 33), "grow": 100, "steps": 10 * rng.randrange(1, 4)}
    if kind == "reduce":
        return {"kind": "reduce", "records": int(_log(rng, 40.0, 65536.0)), "key_bits": rng.randrange(20, 41),
                "per_key": round(_log(rng, 1.0, 50.0), 2)}
    return {"kind": "colocation", "excitors": int(_log(rng, 100.0, 5000.0)), "orbitals": rng.choice([66, 114, 186, 358]),
            "processors": int(_log(rng, 2.0, 1000.0)), "move": rng.randrange(0, 8),
            "iterations": int(_log(rng, 64.0, 4096.0)), "checkpoints": rng.randrange(1, 12)}


# -- one wavefunction ------------------------------------------------------


@functools.lru_cache(maxsize=1)
def _integrals():
    return molecule_integrals(norb=41, nocc=10, seed=7)


def _room(case, population):
    """List entries to make room for: the whole space, or the overshoot of a growing population."""
    if case["system"] == "gas" and (case["orbitals"], case["level"]) in SATURATED:
        return SATURATED[case["orbitals"], case["level"]] + 65536
    return int(4 * population) + 65536


def _context(case, stream, population, **run):
    more = {}
    if case["system"] == "molecule":
        more["h1"], more["eri"] = _integrals()
    return ccmc.Context("ueg" if case["system"] == "gas" else "generic", case["electrons"], case["orbitals"],
                        case["level"], rs=case["rs"], target_pop=population, precision=case["precision"],
                        stream=stream.cuda_stream, list_capacity=_room(case, population), **run, **more)


def _host(shape):
    """A page-locked host array, as a program that moves lists every few steps keeps."""
    return torch.zeros(shape, dtype=torch.int64, pin_memory=True).numpy()


def _restart_point(ctx, population=None):
    """The context's list (scaled to a population) and run state, in host memory of the program's own."""
    bits, _, pop = ctx.get_list(with_keys=False)
    it, shift, _, _ = ctx.get_state()
    if population is not None:
        scale = population * 65536.0 / float(np.abs(pop).sum(dtype=np.float64))
        # every occupied excitor holds at least one particle
        mag = np.maximum(np.rint(np.abs(pop) * scale).astype(np.int64), 65536)
        pop = np.where(pop < 0, -mag, mag)
    n_total = float(np.abs(pop).sum(dtype=np.float64)) / 65536.0
    hb, hp = _host(bits.shape), _host(pop.shape)
    hb[:] = bits.view(np.int64)
    hp[:] = pop
    return hb.view(np.uint64), hp, it, shift, n_total


def _prepare_steps(case, seed):
    stream = torch.cuda.Stream()
    population, gas = case["population"], case["system"] == "gas"
    ctx = _context(case, stream, population, tau=case["tau"], fnc=case["sampler"] != "original",
                   multispawn=case["sampler"] == "multispawn", seed=seed + 1, n_ranks=case["processors"],
                   nu_move=case["move"])
    # the original sampler fills a list fastest; a saturated list is grown at a smaller population and scaled up
    saturates = gas and (case["orbitals"], case["level"]) in SATURATED
    grown_at = min(population, 1.0e6) if saturates else population
    share = 0.15 if gas and case["rs"] <= 2.0 else 0.05
    many = case["sampler"] == "multispawn"
    with_one = _context(case, stream, grown_at, tau=(0.01 if saturates else case["tau"]) if gas else 1.0e-5,
                        seed=seed + 1001, fnc=many and not saturates, multispawn=many and not saturates,
                        d0_init=share * grown_at * (1.0 + 0.01 * (seed % 7)))
    for _ in range(200):
        with_one.step(2)
        if with_one.energy()["n_total"] >= grown_at:
            break
    bits, pop, it, shift, n_total = _restart_point(with_one, population)
    with_one.close()
    # a list has at most one excitor per particle; rows beyond its end stay zero
    room = min(_room(case, population), (int(1.25 * population) if not gas else 4 * int(population)) + 65536)
    out = (_host((room, ctx.nw)).view(np.uint64), _host(room).view(np.uint64), _host(room))
    return {"case": case, "stream": stream, "ctx": ctx, "bits": bits, "pop": pop, "it": it, "shift": shift,
            "n_total": n_total, "out": out}


def _records(recs):
    """The per-step records as (whole numbers, floating numbers)."""
    whole = [k for k in recs[0] if k not in ("shift", "e_num")]
    return (np.array([[r[k] for k in whole] for r in recs], dtype=np.int64),
            np.array([[r["shift"], r["e_num"]] for r in recs], dtype=np.float64))


def _run_steps(s):
    ctx = s["ctx"]
    ctx.set_state(s["it"], s["shift"], True, s["n_total"])
    ctx.set_list(s["bits"], s["pop"])
    ctx.step(s["case"]["steps"])
    energy = ctx.energy()
    whole, floating = _records(ctx.records(s["case"]["steps"]))
    _, _, pop = ctx.get_list(out=s["out"])
    return {"bits": s["out"][0].view(np.int64), "keys": s["out"][1].view(np.int64), "pop": s["out"][2],
            "excitors": len(pop), "records": whole, "estimators": floating, "e_proj": energy["e_proj"]}


# -- many wavefunctions ----------------------------------------------------


def _prepare_batch(case, seed):
    stream = torch.cuda.Stream()
    ctxs, targets = [], []
    for w in batched_replicas(case["replicas"]):
        targets.append(w["target_pop"])
        w.update(seed=w["seed"] + 101 * seed, d0_init=0.2 * w["target_pop"], tau=0.005,
                 list_capacity=int(2 * w["target_pop"]) + 65536, spawn_capacity=int(4 * w["target_pop"]) + 65536)
        ctxs.append(ccmc.from_workload(w, stream=stream.cuda_stream))
    batch = ccmc.Batch(ctxs, stream.cuda_stream)
    batch.step(case["grow"])
    starts = [_restart_point(c, t) for c, t in zip(ctxs, targets)]
    rooms = [2 * int(t) + 65536 for t in targets]
    rooms = [min(r, SATURATED[c.nso, c.lmax]) for r, c in zip(rooms, ctxs)]
    return {"case": case, "stream": stream, "batch": batch, "ctxs": ctxs, "starts": starts,
            "bits": _host(sum(r * c.nw for r, c in zip(rooms, ctxs))).view(np.uint64), "pop": _host(sum(rooms))}


def _run_batch(s):
    for c, (bits, pop, it, shift, n_total) in zip(s["ctxs"], s["starts"]):
        c.set_state(it, shift, True, n_total)
        c.set_list(bits, pop)
    s["batch"].step(s["case"]["steps"])
    b = p = 0
    energies, sizes = [], []
    for c in s["ctxs"]:
        energies.append(list(c.energy().values()))
        n = c.list_size()
        # the lists one after another in the program's two buffers
        c.get_list(out=(s["bits"][b : b + n * c.nw].reshape(n, c.nw), None, s["pop"][p : p + n]), with_keys=False)
        sizes.append(n)
        b += n * c.nw
        p += n
    return {"sizes": np.array(sizes, dtype=np.int64), "bits": s["bits"].view(np.int64), "pop": s["pop"],
            "energies": np.array(energies, dtype=np.float64)}


# -- standalone calls ------------------------------------------------------


def _prepare_reduce(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    n = case["records"]
    distinct = max(1, int(n / case["per_key"]))
    # distinct keys spread over the key range, each held by n / distinct records on average, in random order
    stride = (1 << case["key_bits"]) // distinct
    pool = torch.arange(distinct, device="cuda") * stride
    pool = pool + torch.randint(0, stride, (distinct,), generator=gen, device="cuda")
    owner = torch.cat([torch.arange(distinct, device="cuda"),
                       torch.randint(0, distinct, (n - distinct,), generator=gen, device="cuda")])
    keys = pool[owner[torch.randperm(n, generator=gen, device="cuda")]]
    pops = torch.randint(-(1 << 18), 1 << 18, (n,), generator=gen, device="cuda")
    return {"case": case, "lib": ccmc.load(), "keys": keys, "pops": pops, "keys_out": torch.empty_like(keys),
            "pops_out": torch.empty_like(pops)}


def _run_reduce(s):
    count = ctypes.c_size_t(0)
    status = s["lib"].ccmc_reduce_records_noalloc(
        s["keys"].data_ptr(), s["pops"].data_ptr(), s["case"]["records"], s["case"]["key_bits"],
        s["keys_out"].data_ptr(), s["pops_out"].data_ptr(), ctypes.byref(count),
        torch.cuda.current_stream().cuda_stream)
    if status:
        raise RuntimeError(f"ccmc_reduce_records_noalloc: status {status}")
    return {"keys": s["keys_out"][: count.value], "pops": s["pops_out"][: count.value]}


def _prepare_colocation(case, seed):
    rng = np.random.default_rng(seed)
    n, m = case["excitors"], case["orbitals"]
    # n determinants of 14 electrons among the orbitals (the reference's with two moved up)
    words = np.zeros((n, (m + 63) // 64), dtype=np.uint64)
    words[:, 0] = (1 << 14) - 1
    holes = np.argsort(rng.random((n, 14)), axis=1)[:, :2]
    parts = 14 + np.argsort(rng.random((n, m - 14)), axis=1)[:, :2]
    for col in np.concatenate([holes, parts], axis=1).T:
        words[np.arange(n), col // 64] ^= np.left_shift(np.uint64(1), (col % 64).astype(np.uint64))
    t, k = case["iterations"], case["checkpoints"]
    checks = sorted({max(1, int(round(t ** ((i + 1) / k)))) for i in range(k)} | {t})
    return {"case": case, "words": words, "checks": checks}


def _run_colocation(s):
    c = s["case"]
    s1, s2 = ccmc.colocation(s["words"], c["processors"], c["move"], s["checks"])
    return {"sum": s1.view(np.int64), "squares": s2.view(np.int64)}


_PREPARE = {"steps": _prepare_steps, "batch": _prepare_batch, "reduce": _prepare_reduce,
            "colocation": _prepare_colocation}
_RUN = {"steps": _run_steps, "batch": _run_batch, "reduce": _run_reduce, "colocation": _run_colocation}


def prepare(case, seed):
    state = _PREPARE[case["kind"]](case, seed)
    state["run"] = _RUN[case["kind"]]
    return state


def run(state):
    return state["run"](state)


# -- what a pass cannot do without -----------------------------------------


def _steps_work(orbitals, level, population, steps, excitors):
    words = (orbitals + 63) // 64
    entry = 8 * words + 16
    # the list read and written once a step; a record of 16 bytes for a tenth of the samples
    bytes_step = 2 * excitors * entry + 1.6 * population
    # two draws of ten Philox rounds (about ten 64-bit operations each) a sample
    return {"bytes": steps * bytes_step + 2 * excitors * entry, "flops": 200.0 * population * steps}


def work(case):
    if case["kind"] == "steps":
        most = SATURATED.get((case["orbitals"], case["level"])) if case["system"] == "gas" else None
        excitors = min(0.7 * case["population"], most or math.inf)
        return _steps_work(case["orbitals"], case["level"], case["population"], case["steps"], excitors)
    if case["kind"] == "batch":
        total = {"bytes": 0.0, "flops": 0.0}
        for w in batched_replicas(case["replicas"]):
            part = _steps_work(w["nso"], w["lmax"], w["target_pop"], case["steps"],
                               min(0.7 * w["target_pop"], SATURATED[w["nso"], w["lmax"]]))
            total = {k: total[k] + part[k] for k in total}
        return total
    if case["kind"] == "reduce":
        n = case["records"]
        return {"bytes": 16.0 * n * (1.0 + 1.0 / case["per_key"]), "flops": n * math.log2(n)}
    # two owners compared and counted per pair and iteration
    n, t = case["excitors"], case["iterations"]
    return {"bytes": 8.0 * n * ((case["orbitals"] + 63) // 64), "flops": 2.0 * t * n * (n - 1) / 2}


def exact(case, seed):
    # whole numbers but for the projected energy, whose terms only the step itself can list
    return None
