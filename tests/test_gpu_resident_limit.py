"""The mailbox wait limit of resident launches: neighbours that answer are waited for however short it
is, as the clock also runs while the GPU does something else; one that never sends ends the wait."""
import time

import pytest

from gpu_util import assert_same, gpu_run, oracle_for
from paper_2405_03605_gb300.workloads import RunShape

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,cols,S", [(32, 32, 64), (40, 41, 256)])
def test_short_limit_waits_for_neighbours_that_answer(rows, cols, S):
    shape = RunShape(rows=rows, cols=cols, surface_sites=S, seed=71)
    g = gpu_run(shape)
    g.resident_policy(0, 1)  # GA_RESIDENT_AUTO, a limit of one microsecond
    g.step(300)
    g.sync()
    assert g.launches == 3
    o = oracle_for(shape)
    o.step(300)
    assert_same(g.snapshot(), o.snapshot(), 32)


def test_short_limit_ends_a_wait_for_nothing():
    from paper_2405_03605_gb300 import ga
    g = gpu_run(RunShape(rows=16, cols=16, seed=72))
    g.resident_policy(2, 1)
    g.inject_lost_migrants(9)
    t0 = time.perf_counter()
    g.step(200)
    with pytest.raises(ga.GaError) as e:
        g.sync()
    assert e.value.code == -4
    assert time.perf_counter() - t0 < 0.5
