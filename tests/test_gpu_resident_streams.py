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


def test_large_runs_stream_beside_a_resident_one():
    """A run that takes the whole GPU when it steps resident streams while another such run does on
    another stream, and steps resident again when that one is done; one captured into a graph neither
    asks nor is counted."""
    import torch
    from paper_2405_03605_gb300 import ga
    shapes = [RunShape(rows=96, cols=97, seed=7, run_id=i) for i in range(3)]
    runs = [ga.Run(s, stream=torch.cuda.Stream()) for s in shapes]
    for r in runs:
        r.sync()
    runs[0].step(12000)  # some 30 ms
    runs[1].step(30)
    assert runs[0].launches == 1 + 3 * 2 and runs[1].launches == 2 + 30
    runs[0].sync()
    runs[1].step(30)
    assert runs[1].launches == 2 + 30 + 2
    runs[1].step(10)  # its own launches do not count
    assert runs[1].launches == 2 + 30 + 4
    runs[1].sync()
    runs[2].step(20)
    runs[2].sync()
    graph = torch.cuda.CUDAGraph()
    before = runs[2].launches
    runs[0].step(4000)
    with torch.cuda.graph(graph, stream=runs[2].stream):
        runs[2].step(20)
    assert runs[2].launches == before + 2
    graph.replay()
    torch.cuda.synchronize()
    for r in runs:
        r.sync()
    assert_same(runs[1].snapshot(), streamed(shapes[1], 70), 32)
    assert_same(runs[2].snapshot(), streamed(shapes[2], 40), 32)
    assert_same(runs[0].snapshot(), streamed(shapes[0], 16000), 32)
    runs[0].step(2000)
    runs[0].close()  # with its launch in flight
    runs[1].step(5)
    runs[1].sync()


def test_runs_of_several_threads():
    """Handles of their own in threads of their own, large enough to fill the GPU resident."""
    import threading

    import torch
    from paper_2405_03605_gb300 import ga
    shapes = [RunShape(rows=96, cols=98, seed=9, run_id=i) for i in range(4)]
    runs = [ga.Run(s, stream=torch.cuda.Stream()) for s in shapes]
    failed = []

    def work(r):
        try:
            for _ in range(12):
                r.step(10)
                r.sync()
        except Exception as e:
            failed.append(e)

    threads = [threading.Thread(target=work, args=(r,)) for r in runs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
    for r, s in zip(runs, shapes):
        assert_same(r.snapshot(), streamed(s, 120), 32)
