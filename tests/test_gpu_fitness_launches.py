"""The float model streamed with launches of many generations, on either side of the lengths at which
its kernel draws the mutations in place instead of queueing them, against the oracle."""
import pytest

from gpu_util import assert_same, gpu_run, oracle_for
from paper_2405_03605_gb300.workloads import RunShape, MODEL_FITNESS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,tsize", [(16, 5), (16, 3), (32, 5), (32, 8), (64, 5), (64, 2)])
@pytest.mark.parametrize("every", [3, 4, 5, 6, 7, 8, 15, 16, 31, 32, 0])
def test_long_launches(N, tsize, every):
    shape = RunShape(rows=3, cols=7, island_size=N, tournament_size=tsize, p_ben=0.003, p_del=0.33,
                     model=MODEL_FITNESS, effect_scale=0.5, migrate_every=every, seed=12 + N + tsize)
    g = gpu_run(shape)
    g.resident_policy(1)  # GA_RESIDENT_OFF
    g.step(2 * every + 17)
    g.sync()
    o = oracle_for(shape)
    o.step(2 * every + 17)
    assert_same(g.snapshot(), o.snapshot(), N)
