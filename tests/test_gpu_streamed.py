"""The streamed kernels against the oracle.  The default policy steps most small synchronous runs
resident, so each shape here is stepped under GA_RESIDENT_OFF, and under the default policy too: every
island size, record size, tournament form and migration interval, blocks with one unit to all of
them, and missing last islands."""
import pytest

from gpu_util import assert_same, gpu_run, oracle_for
from paper_2405_03605_gb300.workloads import RunShape, variant_shapes, STEADY, TILTED, HYBRID

pytestmark = pytest.mark.gpu

AUTO, OFF = 0, 1


def check(shape, gens, chunks=None):
    o = oracle_for(shape)
    o.step(gens)
    expected = o.snapshot()
    for mode in (OFF, AUTO):
        g = gpu_run(shape)
        g.resident_policy(mode)
        for c in (chunks or [gens]):
            g.step(c)
        g.sync()
        assert_same(g.snapshot(), expected, shape.island_size)


# units of the streamed kernel: 16 islands of 16, 8 of 32 or of 64; four or eight units to a block
@pytest.mark.parametrize("every", [1, 2, 16, 0])
@pytest.mark.parametrize("tsize", [5, 3])
@pytest.mark.parametrize("N,rows,cols", [
    (16, 1, 1), (16, 3, 5), (16, 1, 17), (16, 7, 9), (16, 8, 8), (16, 5, 13), (16, 11, 13),
    (32, 1, 1), (32, 1, 7), (32, 3, 3), (32, 5, 7), (32, 7, 9), (32, 8, 8), (32, 5, 13), (32, 11, 13),
    (64, 1, 7), (64, 3, 3), (64, 5, 7), (64, 7, 9), (64, 5, 13),
])
def test_units(N, rows, cols, tsize, every):
    check(RunShape(rows=rows, cols=cols, island_size=N, tournament_size=tsize, migrate_every=every,
                   seed=11 + N + rows, run_id=cols, p_ben=0.05, p_del=0.05), 70)


@pytest.mark.parametrize("N,rows,cols", [(4, 5, 7), (8, 7, 9), (16, 9, 11), (32, 13, 17), (64, 6, 10),
                                         (128, 5, 3)])
def test_island_sizes(N, rows, cols):
    check(RunShape(rows=rows, cols=cols, island_size=N, seed=1234 + N, run_id=N), 150)


@pytest.mark.parametrize("n", [1, 2, 3, 4, 6, 7, 8])
@pytest.mark.parametrize("N", [8, 16, 64])
def test_tournament_sizes(N, n):
    check(RunShape(rows=6, cols=5, island_size=N, tournament_size=n, p_ben=0.05, p_del=0.05, seed=n), 80)


@pytest.mark.parametrize("name", ["steady256x1", "tilted32x8", "hybrid64x1"])
@pytest.mark.parametrize("N", [8, 16, 32, 64])
@pytest.mark.parametrize("k", [1, 4, 16])
def test_surface_variants(name, N, k):
    check(variant_shapes(N, migrate_every=k)[name].with_(rows=max(2, 8 * 32 // N), cols=7), 130)


@pytest.mark.parametrize("S,b,policy", [(128, 1, STEADY), (16, 2, STEADY), (8, 4, STEADY), (4, 1, STEADY),
                                        (64, 4, TILTED), (32, 1, HYBRID), (16, 8, TILTED), (8, 1, HYBRID)])
@pytest.mark.parametrize("N", [16, 32])
def test_more_surfaces(N, S, b, policy):
    check(RunShape(rows=4, cols=9, island_size=N, surface_sites=S, differentia_bits=b, curation=policy,
                   seed=S * 10 + b), 200)


@pytest.mark.parametrize("rows,cols", [(1, 1), (1, 5), (4, 1), (2, 2), (3, 2)])
@pytest.mark.parametrize("S", [64, 128, 256])
def test_degenerate_tori(rows, cols, S):
    check(RunShape(rows=rows, cols=cols, surface_sites=S, seed=rows * 100 + cols), 60)


def test_launches_of_256_generations():
    shape = RunShape(rows=5, cols=6, migrate_every=0, seed=77)
    g = gpu_run(shape)
    g.resident_policy(OFF)
    g.step(600)
    g.sync()
    assert g.launches == 2 + 3  # founder, site table, three launches of at most 256 generations
    o = oracle_for(shape)
    o.step(600)
    assert_same(g.snapshot(), o.snapshot(), 32)
    check(shape, 600, chunks=[1, 299, 300])


@pytest.mark.parametrize("p_ben,p_del", [(0.0, 0.0), (1.0, 0.0), (0.0, 1.0), (0.5, 0.5), (1e-4, 1e-1)])
def test_mutation_extremes(p_ben, p_del):
    check(RunShape(rows=4, cols=4, p_ben=p_ben, p_del=p_del, seed=5), 64)


@pytest.mark.parametrize("n_gens,launches", [(3, 1 + 1 + 3), (4, 3)])
def test_auto_generations(n_gens, launches):
    """Runs without mailboxes in their workspace stream in calls of fewer than four generations."""
    shape = RunShape(rows=6, cols=7, surface_sites=256, seed=6)
    g = gpu_run(shape)
    g.step(n_gens)
    g.sync()
    assert g.launches == launches
    o = oracle_for(shape)
    o.step(n_gens)
    assert_same(g.snapshot(), o.snapshot(), 32)


# 48-byte records leave through shared memory up to one generation to a launch (four in islands of
# more than 32) or 32,768 islands, else directly; blocks with missing last islands
@pytest.mark.parametrize("N,rows,cols,every", [(32, 181, 182, 1), (32, 181, 182, 2), (64, 181, 183, 4), (64, 181, 183, 5),
                                               (32, 181, 181, 2), (128, 3, 5, 4), (128, 3, 5, 5)])
def test_48_byte_stores(N, rows, cols, every):
    shape = RunShape(rows=rows, cols=cols, island_size=N, surface_sites=256, migrate_every=every, seed=8 + N)
    g = gpu_run(shape)
    g.resident_policy(OFF)
    g.step(2 * every + 1)
    g.sync()
    o = oracle_for(shape)
    o.step(2 * every + 1)
    assert_same(g.snapshot(), o.snapshot(), N)


@pytest.mark.parametrize("N,rows,cols,S,b,policy", [(64, 3, 5, 64, 1, STEADY), (64, 2, 3, 256, 1, HYBRID), (64, 3, 3, 32, 4, TILTED),
                                                    (128, 2, 3, 64, 1, STEADY), (128, 3, 3, 128, 1, HYBRID),
                                                    (128, 2, 2, 32, 8, TILTED), (16, 3, 5, 256, 1, STEADY)])
@pytest.mark.parametrize("every", [1, 4])
def test_mixed_counters(N, rows, cols, S, b, policy, every):
    """Loaded populations whose agents' counters differ, in islands whose traits and surfaces are looked
    up in shared memory: every agent's deposit follows its own counter."""
    shape = RunShape(rows=rows, cols=cols, island_size=N, surface_sites=S, differentia_bits=b, curation=policy,
                     migrate_every=every, seed=21 + N)
    src = oracle_for(shape.with_(migrate_every=1))
    src.step_async(60, window=7)
    mixed = src.snapshot()
    o = oracle_for(shape)
    o.load(mixed, 60)
    o.step(35)
    g = gpu_run(shape)
    g.load(mixed, 60)
    g.step(35)
    g.sync()
    assert_same(g.snapshot(), o.snapshot(), N)
