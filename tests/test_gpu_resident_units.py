"""Resident launches whose warps hold several islands (more than eight: a second round of mailbox
reads), for every record size and both genome models, and the runs that stream, against the oracle."""
import pytest

from gpu_util import assert_same, gpu_run, oracle_for
from paper_2405_03605_gb300.workloads import RunShape, MODEL_FITNESS, MODEL_TRAIT

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,rows,cols,S,every,tsize,model,gens", [
    (32, 170, 171, 128, 1, 3, MODEL_TRAIT, 14),   # eleven islands to a warp
    (16, 200, 199, 128, 1, 5, MODEL_TRAIT, 14),   # sixteen to a warp, the last one short
    (32, 71, 83, 256, 1, 5, MODEL_TRAIT, 60),
    (32, 97, 98, 256, 2, 3, MODEL_TRAIT, 40),
    (64, 61, 97, 256, 1, 5, MODEL_TRAIT, 40),
    (16, 111, 113, 256, 1, 8, MODEL_TRAIT, 40),
    (32, 40, 76, 64, 1, 3, MODEL_TRAIT, 40),      # 3,040 islands: the last size of one to a warp
    (32, 1, 3041, 64, 1, 3, MODEL_TRAIT, 40),
    (32, 50, 52, 64, 1, 5, MODEL_TRAIT, 40),      # two to a warp from 2,433 on
    (32, 60, 61, 64, 1, 5, MODEL_FITNESS, 40),
    (32, 60, 61, 64, 4, 3, MODEL_FITNESS, 40),
    (16, 91, 90, 64, 4, 3, MODEL_FITNESS, 40),    # a pair of islands to a warp, 27 warps on an SM
    (16, 130, 99, 64, 1, 5, MODEL_FITNESS, 40),
    (64, 57, 61, 64, 16, 5, MODEL_FITNESS, 40),
])
def test_several_islands_to_a_warp(N, rows, cols, S, every, tsize, model, gens):
    shape = RunShape(rows=rows, cols=cols, island_size=N, tournament_size=tsize, surface_sites=S,
                     migrate_every=every, model=model, seed=900 + N + S, run_id=rows, p_ben=0.05,
                     p_del=0.33 if model else 0.05)
    g = gpu_run(shape)
    g.step(gens)
    g.sync()
    assert g.launches == 3  # founder, set-up, one resident launch
    o = oracle_for(shape)
    o.step(gens)
    assert_same(g.snapshot(), o.snapshot(), N)


@pytest.mark.parametrize("N,rows,cols,S,every,model,launches", [
    (16, 200, 203, 256, 1, MODEL_TRAIT, 3), (16, 205, 210, 256, 1, MODEL_TRAIT, 2 + 8),
    (16, 290, 210, 128, 1, MODEL_TRAIT, 2 + 8), (16, 64, 65, 128, 4, MODEL_TRAIT, 2 + 2),
    (32, 140, 141, 64, 1, MODEL_FITNESS, 3), (32, 150, 151, 64, 1, MODEL_FITNESS, 2 + 8),
    (64, 25, 41, 128, 8, MODEL_TRAIT, 2 + 1), (8, 110, 110, 256, 1, MODEL_TRAIT, 3),
])
def test_auto_streams_where_that_is_faster(N, rows, cols, S, every, model, launches):
    """GA_RESIDENT_AUTO by record size and migration interval: a founder, a set-up or site table, and
    one resident launch or one for each migration interval; both give the oracle's result."""
    shape = RunShape(rows=rows, cols=cols, island_size=N, surface_sites=S, migrate_every=every, model=model,
                     seed=50 + N + S, p_ben=0.05, p_del=0.33 if model else 0.05)
    g = gpu_run(shape)
    g.step(8)
    g.sync()
    assert g.launches == launches
    o = oracle_for(shape)
    o.step(8)
    assert_same(g.snapshot(), o.snapshot(), N)
