"""Performance cases: the work a user of the library has it do, through its public binding.

Three kinds of call carry real use.  "step": a GA run brought from its founders to a
generation count and its population read out (the paper's experiment and one served request
are both this).  "batch": heterogeneous replicate runs advanced together by shared launches.
"mrca": pairwise MRCA bounds over sampled end-state agents, for synchronous runs (one counter)
and asynchronous ones (agents' counters differ).  Free-running asynchronous stepping is left
out: its outputs depend on scheduling, so two passes on the same inputs do not agree; its
post hoc analysis is here, on a population grown by the reproducible asynchronous schedule.

Outputs are whole populations (as 32-bit words) and whole (lo, hi) arrays: integers and bytes
throughout, reproducible bit for bit.
"""
import math

import torch

from paper_2405_03605_gb300 import ga
from paper_2405_03605_gb300.workloads import (
    ASYNC, ASYNC_SEQUENTIAL, HYBRID, MODEL_FITNESS, MODEL_TRAIT, STEADY, SYNC, TILTED, RunShape,
    batch_shapes, sample_agent_ids)

# Populations up to this size can stay on the chip (registers and shared memory of 152 SMs), so
# only their first read and last write are unavoidable; larger ones stream through device
# memory once per migration interval.
ON_CHIP_BYTES = 30e6

# 32-bit operations of one birth: ten Philox rounds of two products (low and high halves) and
# two three-input XORs, then tournament, copy, mutation and deposit; and of one normal deviate
# of the float model (a second Philox call and Box-Muller).
BIRTH_OPS = 10 * 6 + 30
DEVIATE_OPS = 10 * 6 + 120
PAIR_OPS = 12


def _step(name, rows, cols, generations, island_size=32, tournament_size=5, p_ben=0.01, p_del=0.01,
          sites=64, bits=1, curation=STEADY, every=1, model=MODEL_TRAIT):
    case = {"kind": "step", "rows": rows, "cols": cols, "island_size": island_size,
            "tournament_size": tournament_size, "p_ben": p_ben, "p_del": p_del, "sites": sites,
            "bits": bits, "curation": curation, "every": every, "model": model,
            "generations": generations}
    return {"name": name, **case} if name else case


def _mrca(name, rows, cols, sample, generations, island_size=32, p_ben=0.01, sites=64, bits=1,
          curation=STEADY, mixed=False, window=1):
    case = {"kind": "mrca", "rows": rows, "cols": cols, "island_size": island_size,
            "tournament_size": 5, "p_ben": p_ben, "p_del": 0.01, "sites": sites, "bits": bits,
            "curation": curation, "every": 1, "model": MODEL_TRAIT, "generations": generations,
            "sample": sample, "mixed": mixed, "window": window}
    return {"name": name, **case} if name else case


def listed():
    return [
        # the smallest served request: about 10,000 agents for 100 generations, where launches
        # and latency count
        _step("request_small", 17, 18, 100),
        # the 32x32 torus of 32-agent islands, 1,000 generations
        _step("torus_32x32", 32, 32, 1000),
        # a served request from the middle of the range, on a ragged torus
        _step("request_mid", 97, 103, 250),
        # the same with 256 retention sites (half of all served requests): 48-byte records
        _step("request_mid_wide", 71, 83, 250, sites=256),
        # the paper-scale grid, 16.8M agents, adaptive treatment
        _step("paper_adaptive", 512, 1024, 100),
        # the paper's own float-fitness treatment on that grid
        _step("paper_fitness", 512, 1024, 50, p_ben=0.003, p_del=0.33, model=MODEL_FITNESS),
        # 4.2M agents with 256 one-bit sites: 48-byte records, migration every generation
        _step("steady256x1", 128, 1024, 100, sites=256),
        # 4.2M agents in islands of 64, 32 eight-bit sites, migration every 16 generations
        _step("tilted32x8_every16", 64, 1024, 160, island_size=64, sites=32, bits=8,
              curation=TILTED, every=16),
        # replicate runs of mixed shape, rates and tournament size advanced together
        {"name": "batch_mix", "kind": "batch", "runs": 32, "mix": 42, "generations": 256},
        # post hoc relatedness of the paper-scale run: 4,096 sampled agents, 8.4M pairs
        _mrca("mrca_sample", 512, 1024, 4096, 1000),
        # the same for a run with 256 sites (strings wider than 64 bits), a ragged sample
        _mrca("mrca_wide", 128, 1024, 3000, 1000, sites=256),
        # the same for an asynchronous run, whose agents carry different counters
        _mrca("mrca_mixed", 8, 16, 3001, 768, mixed=True, window=64),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


# record layouts users choose: (sites, bits, curation)
_SURFACES = [(64, 1, STEADY), (64, 1, STEADY), (256, 1, STEADY), (32, 8, TILTED), (64, 1, HYBRID),
             (128, 1, STEADY), (32, 2, STEADY), (16, 4, TILTED)]


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "batch", "mrca", "mrca"])
    if kind == "batch":
        return {"kind": "batch", "runs": rng.randint(4, 32), "mix": rng.randrange(1, 1 << 20),
                "generations": rng.randint(64, 128)}
    sites, bits, curation = rng.choice(_SURFACES)
    if kind == "mrca":
        sample = int(_log_uniform(rng, 64, 4096))
        if rng.random() < 0.4:
            return _mrca(None, rng.randint(8, 12), rng.randint(11, 16), min(sample, 2816),
                         rng.randint(200, 700), sites=sites, bits=bits, curation=curation, mixed=True,
                         window=rng.choice([16, 64]))
        return _mrca(None, rng.randint(100, 400), rng.randint(200, 700), sample,
                     rng.randint(200, 1000), island_size=rng.choice([16, 32, 64]),
                     p_ben=rng.choice([0.0, 0.01]), sites=sites, bits=bits, curation=curation)
    island_size = rng.choice([8, 16, 32, 32, 32, 64, 128])
    model, p_ben, p_del = MODEL_TRAIT, _log_uniform(rng, 1e-4, 1e-1), _log_uniform(rng, 1e-4, 1e-1)
    if island_size in (16, 32, 64) and rng.random() < 0.25:
        model, p_ben, p_del, sites, bits, curation = MODEL_FITNESS, 0.003, 0.33, 64, 1, STEADY
    agents = _log_uniform(rng, 1e4, 1e7)
    islands = max(4, round(agents / island_size))
    rows = max(2, round(math.sqrt(islands) * rng.uniform(0.5, 1.5)))
    cols = max(2, islands // rows)
    agents = rows * cols * island_size
    gens = max(20, min(int(_log_uniform(rng, 100, 1000)), int(4e8 / agents)))
    return _step(None, rows, cols, gens, island_size, rng.choice([5, 5, 5, 2, 3, 4, 6, 7, 8]),
                 p_ben, p_del, sites, bits, curation, rng.choice([1, 1, 1, 4, 16]), model)


def _shape(case, seed, mode=SYNC):
    return RunShape(rows=case["rows"], cols=case["cols"], island_size=case["island_size"],
                    tournament_size=case["tournament_size"], p_ben=case["p_ben"],
                    p_del=case["p_del"], surface_sites=case["sites"],
                    differentia_bits=case["bits"], curation=case["curation"],
                    migrate_every=case["every"], seed=(seed * 0x9E3779B97F4A7C15) % (1 << 64),
                    run_id=seed % 1000, generations=case["generations"], model=case["model"],
                    mode=mode, async_window=case.get("window", 1) if mode != SYNC else 1)


def _mix(case, seed):
    return [s.with_(seed=(seed * 0x9E3779B97F4A7C15) % (1 << 64))
            for s in batch_shapes(case["runs"], seed=case["mix"], generations=case["generations"])]


def _output(run):
    return torch.empty((run.n_agents, run.record_bytes), dtype=torch.uint8, device="cuda")


def prepare(case, seed):
    if case["kind"] == "step":
        run = ga.Run(_shape(case, seed))
        return {"kind": "step", "run": run, "generations": case["generations"], "out": _output(run)}
    if case["kind"] == "batch":
        # members and batch share a stream, so a pass's read-outs precede the next pass's steps
        stream = torch.cuda.Stream()
        runs = [ga.Run(s, stream=stream) for s in _mix(case, seed)]
        return {"kind": "batch", "runs": runs, "batch": ga.Batch(runs, stream=stream),
                "generations": case["generations"], "outs": [_output(r) for r in runs]}
    if case["mixed"]:
        # an asynchronous population grown by the reproducible schedule, in a run of the
        # free-running mode
        grown = ga.Run(_shape(case, seed, ASYNC_SEQUENTIAL))
        grown.step(case["generations"])
        records = grown.snapshot()
        grown.close()
        run = ga.Run(_shape(case, seed, ASYNC))
        run.load(records, case["generations"])
    else:
        run = ga.Run(_shape(case, seed))
        run.step(case["generations"])
        run.sync()
    n = case["sample"]
    ids = torch.from_numpy(sample_agent_ids(run.n_agents, n, seed=seed).astype("int32")).cuda()
    lo, hi = (torch.empty(n * (n - 1) // 2, dtype=torch.int32, device="cuda") for _ in range(2))
    return {"kind": "mrca", "run": run, "ids": ids, "lo": lo, "hi": hi}


def run(state):
    if state["kind"] == "step":
        # one run: founders, the generations, the final population
        r = state["run"]
        r.reset()
        r.step(state["generations"])
        return r.snapshot_device(state["out"]).view(torch.int32)
    if state["kind"] == "batch":
        # one stretch of generations of every member, then every population; each pass goes on
        # from where the last one stopped, as a service does
        state["batch"].step(state["generations"])
        state["batch"].sync()
        return [r.snapshot_device(o).view(torch.int32)
                for r, o in zip(state["runs"], state["outs"])]
    return state["run"].mrca_bounds_device(state["ids"], state["lo"], state["hi"])


def _step_work(shape):
    population = shape.n_agents * shape.record_bytes
    passes = 1 if population <= ON_CHIP_BYTES else -(-shape.generations // max(1, shape.migrate_every))
    ops = BIRTH_OPS
    if shape.model == MODEL_FITNESS:
        ops += DEVIATE_OPS * (shape.p_ben + shape.p_del)
    return 2.0 * population * passes, float(shape.n_agents) * shape.generations * ops


def work(case):
    if case["kind"] == "mrca":
        n = case["sample"]
        pairs = n * (n - 1) // 2
        record = _shape(case, 0).record_bytes
        return {"bytes": n * (4.0 + record) + 8.0 * pairs, "flops": float(PAIR_OPS) * pairs}
    shapes = [_shape(case, 0)] if case["kind"] == "step" else _mix(case, 0)
    each = [_step_work(s) for s in shapes]
    return {"bytes": sum(b for b, _ in each), "flops": sum(f for _, f in each)}


def exact(case, seed):
    """No output here is a rounded number: populations are bytes and the bounds whole numbers, which
    are held equal."""
    return None
