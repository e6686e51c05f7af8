"""Migrants wider than 16 bytes cross in 16-byte chunks, each of which has to arrive whole: many
short resident launches, where what was in the mailboxes before is still unlike any record,
against the streamed kernels."""
import pytest

from gpu_util import assert_same, gpu_run
from paper_2405_03605_gb300.workloads import RunShape

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,rows,cols,S", [(16, 120, 131, 128), (32, 110, 111, 128), (64, 61, 97, 128),
                                           (16, 111, 113, 256), (32, 97, 98, 256), (64, 61, 97, 256)])
def test_migrants_arrive_whole(N, rows, cols, S):
    shape = RunShape(rows=rows, cols=cols, island_size=N, surface_sites=S, seed=31 + N + S)
    ref = gpu_run(shape)
    ref.resident_policy(1)  # GA_RESIDENT_OFF
    ref.step(4)
    ref.sync()
    expected = ref.snapshot()
    g = gpu_run(shape)
    for _ in range(25):
        g.reset()
        before = g.launches
        g.step(4)
        assert g.launches - before == 2  # set-up and one resident launch
        assert_same(g.snapshot(), expected, N)
