"""Worker for tests/test_gpu_device_checks_streamed.py: the device-check build of the library over runs
that stream (GA_RESIDENT_OFF) and the same runs under the default policy.  Each case must finish with
a clean status and the oracle's result."""
import os
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, HERE)
sys.path.insert(0, os.path.dirname(HERE))

import numpy as np  # noqa: E402

from gpu_util import assert_same, oracle_for  # noqa: E402
from paper_2405_03605_gb300 import ga  # noqa: E402
from paper_2405_03605_gb300.workloads import (RunShape, STEADY, TILTED, HYBRID, MODEL_FITNESS,  # noqa: E402
                                              sample_agent_ids)


def case(shape, gens, ids=0, modes=(1, 0)):
    o = oracle_for(shape)
    o.step(gens)
    expected = o.snapshot()
    for mode in modes:
        g = ga.Run(shape)
        g.resident_policy(mode)
        g.step(gens)
        g.sync()
        assert_same(g.snapshot(), expected, shape.island_size)
        if ids:
            sample = sample_agent_ids(shape.n_agents, ids, seed=3)
            lo, hi = g.mrca_bounds(sample)
            g.sync()
            elo, ehi = o.mrca_bounds(sample)
            assert np.array_equal(lo, elo) and np.array_equal(hi, ehi)
        g.close()
    return len(modes)


def main():
    assert os.path.basename(ga.LIB_PATH) == "libga_debug.so", ga.LIB_PATH
    n = 0
    for N, rows, cols in ((8, 3, 9), (16, 4, 5), (16, 11, 13), (32, 6, 7), (32, 7, 11), (64, 3, 4), (64, 5, 13),
                          (128, 2, 3), (32, 1, 1), (16, 1, 5), (32, 4, 1)):
        for S, b, policy in ((64, 1, STEADY), (128, 1, HYBRID), (32, 8, TILTED), (256, 1, STEADY)):
            for every in (1, 3, 0):
                n += case(RunShape(rows=rows, cols=cols, island_size=N, surface_sites=S, differentia_bits=b,
                                   curation=policy, migrate_every=every, seed=N + S, run_id=every,
                                   tournament_size=5 if every else 3), 40)
    for N, rows, cols in ((16, 3, 11), (32, 5, 13), (64, 3, 7)):
        for tsize in (5, 3):
            for every in (1, 3, 20):
                n += case(RunShape(rows=rows, cols=cols, island_size=N, tournament_size=tsize, migrate_every=every,
                                   model=MODEL_FITNESS, p_ben=0.003, p_del=0.33, seed=N + tsize), 40)
    # resident without mailboxes in the workspace, several islands to a warp
    for N, rows, cols, S, every in ((32, 91, 101, 64, 1), (32, 97, 98, 256, 1), (16, 120, 131, 128, 1), (8, 93, 95, 64, 1)):
        n += case(RunShape(rows=rows, cols=cols, island_size=N, surface_sites=S, migrate_every=every, seed=N), 8, modes=(0,))
    # samples of several blocks of the packing kernel, narrow and wide
    for S in (64, 256):
        n += case(RunShape(rows=16, cols=24, surface_sites=S, seed=S), 100, ids=777)
    print(f"device checks clean over {n} cases")


if __name__ == "__main__":
    main()
