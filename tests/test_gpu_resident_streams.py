"""Several runs stepping at once on several streams, under the default policy: same results as streamed
one by one."""
import pytest

from gpu_util import assert_same, gpu_run
from paper_2405_03605_gb300.workloads import RunShape, MODEL_FITNESS, MODEL_TRAIT

pytestmark = pytest.mark.gpu


def streamed(shape, gens):
    g = gpu_run(shape)
    g.resident_policy(1)  # GA_RESIDENT_OFF
    g.step(gens)
    g.sync()
    return g.snapshot()


@pytest.mark.parametrize("N,rows,cols,S,every,model", [
    (32, 45, 46, 64, 1, MODEL_TRAIT), (32, 45, 46, 64, 1, MODEL_FITNESS), (16, 60, 61, 64, 4, MODEL_TRAIT),
    (64, 31, 33, 64, 1, MODEL_TRAIT), (32, 97, 103, 64, 1, MODEL_TRAIT), (16, 111, 113, 64, 4, MODEL_FITNESS),
    (32, 71, 83, 256, 1, MODEL_TRAIT),
])
def test_runs_at_once(N, rows, cols, S, every, model):
    import torch
    from paper_2405_03605_gb300 import ga
    shapes = [RunShape(rows=rows, cols=cols, island_size=N, surface_sites=S, migrate_every=every, model=model,
                       seed=5 + N, run_id=i, p_del=0.33 if model else 0.05) for i in range(4)]
    runs = [ga.Run(s, stream=torch.cuda.Stream()) for s in shapes]
    for _ in range(3):
        for r in runs:
            r.step(40)
    for r, s in zip(runs, shapes):
        r.sync()
        assert_same(r.snapshot(), streamed(s, 120), N)
