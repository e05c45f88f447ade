"""The band kernel (many steps per launch, the cavity on chip across the GPU, AUTO's
choice for runs of steps of cavities up to about 512^2; small ones in one cluster) against the one-step TMA
kernel: the same bits in every storage mode and rounding, for odd sizes, one and
several rows and passes per block, and every way a run is split into launches."""
import os
import subprocess
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

pytestmark = pytest.mark.gpu

RUNS = (5, 6, 1, 7, 64, 515, 2)  # 515: two launches, the remainder of the first too short for one
MODES = [(0, 0), (1, 0), (1, 1), (2, 0), (2, 1), (3, 0), (3, 1), (4, 0), (4, 1)]
# The last columns: a whole warp of pairs per row, one pair more; rows that fill the
# last block and that leave it one row; 16-bit storage of small cavities; rows wider
# than half a block; several passes per thread.
SIZES = [(128, 128), (130, 127), (193, 305), (64, 97), (33, 304), (640, 151), (512, 512), (380, 307), (8, 600),
         (64, 64), (100, 60), (127, 33), (66, 17), (8, 250)]


def advance(nx, ny, storage, rounding, kernel, walls=(0, 0), cap=4096, runs=RUNS):
    from paper_1601_04633_gb300 import dmrt as D

    p = D.make_params(nx, ny, min(1e4, 0.01 * (12 * ny) ** 2), 0.01, storage=storage, rounding=rounding, kernel=kernel,
                      nu_capacity=cap, left_wall=walls[0], right_wall=walls[1], theta_ref=0.1)
    rng = np.random.default_rng(nx * 10007 + ny)
    sim = D.Cavity2D(p, theta0=0.3 * rng.standard_normal((ny, nx)),
                     theta_hot_profile=0.5 + 0.01 * rng.standard_normal(ny))
    for n in runs:
        sim.step(n)
    sim.check()
    mean, rows, series = sim.nusselt(cap)
    out = [sim.get_state(), rows, series, np.array(mean)] + [t.cpu().numpy() for t in sim.fields()]
    sim.close()
    return out


def assert_same(a, b):
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("storage,rounding", MODES)
@pytest.mark.parametrize("nx,ny", SIZES)
def test_band_equals_single_steps(nx, ny, storage, rounding):
    assert_same(advance(nx, ny, storage, rounding, 0), advance(nx, ny, storage, rounding, 2))


@pytest.mark.parametrize("walls", [(1, 0), (0, 1), (1, 1)])
@pytest.mark.parametrize("storage", [0, 3, 4])
def test_band_wall_kinds(walls, storage):
    assert_same(advance(131, 160, storage, 2, 0, walls), advance(131, 160, storage, 2, 2, walls))


@pytest.mark.parametrize("cap", [1, 3, 100])
def test_band_short_nusselt_ring(cap):
    assert_same(advance(130, 127, 0, 0, 0, cap=cap), advance(130, 127, 0, 0, 2, cap=cap))


def test_band_after_a_checkpoint():
    """Messages left by the steps before a load carry no tag of the steps after it."""
    from paper_1601_04633_gb300 import dmrt as D

    sims = [D.Cavity2D(D.make_params(130, 127, 1e4, 0.01, kernel=k, nu_capacity=64)) for k in (0, 2)]
    for sim in sims:
        sim.step(40)
        blob = sim.save()
        sim.step(40)
        sim.load(blob)
        sim.step(40)
        sim.load(blob)
        sim.step(33)
    np.testing.assert_array_equal(sims[0].get_state(), sims[1].get_state())
    np.testing.assert_array_equal(sims[0].nusselt(64)[2], sims[1].nusselt(64)[2])


def test_band_on_two_streams():
    import torch
    from paper_1601_04633_gb300 import dmrt as D

    ps = [D.make_params(200, 190, 1e4 * (1 + k), 0.01, nu_capacity=512) for k in range(3)]
    sims = [D.Cavity2D(p, stream=torch.cuda.Stream()) for p in ps]
    for _ in range(3):
        for sim in sims:
            sim.step(100)
    for p, sim in zip(ps, sims):
        sim.check()
        ref = D.Cavity2D(D.make_params(200, 190, p.Ra, 0.01, nu_capacity=512, kernel=2))
        ref.step(300)
        np.testing.assert_array_equal(sim.get_state(), ref.get_state())


@pytest.mark.parametrize("sizes", [((300, 290), (130, 127)), ((80, 90), (60, 60))], ids=["band", "cluster"])
def test_a_smaller_context_leaves_a_larger_one_its_shared_memory(sizes):
    from paper_1601_04633_gb300 import dmrt as D

    sims = [D.Cavity2D(D.make_params(nx, ny, 1e3, 0.01, nu_capacity=64)) for nx, ny in sizes]
    for sim in sims:
        sim.step(20)
    for sim, (nx, ny) in zip(sims, sizes):
        ref = D.Cavity2D(D.make_params(nx, ny, 1e3, 0.01, nu_capacity=64, kernel=2))
        ref.step(20)
        np.testing.assert_array_equal(sim.get_state(), ref.get_state())


def test_band_captured_and_replayed():
    """A captured run of an even number of steps goes on from where the last replay ended."""
    import torch
    from paper_1601_04633_gb300 import dmrt as D

    s = torch.cuda.Stream()
    sim = D.Cavity2D(D.make_params(200, 190, 1e4, 0.01, nu_capacity=512), stream=s)
    sim.step(20)
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=s):
        sim.step(20)
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    ref = D.Cavity2D(D.make_params(200, 190, 1e4, 0.01, nu_capacity=512, kernel=2))
    ref.step(80)
    np.testing.assert_array_equal(sim.get_state(), ref.get_state())


def test_band_bounds_checked_build():
    code = ("import sys; sys.path.insert(0, %r); from tests.test_band import advance;"
            "[advance(nx, ny, s, 2, 0) for nx, ny in ((130, 127), (193, 305), (640, 151), (100, 60)) for s in range(5)]" % ROOT)
    subprocess.run([sys.executable, "-c", code], check=True, cwd=ROOT,
                   env=dict(os.environ, DMRT_LIBRARY="bounds_check"))


@pytest.mark.parametrize("storage,rounding", [(0, 0), (1, 1), (4, 0)])
@pytest.mark.parametrize("nx,ny", [(9, 256), (9, 257), (16, 1100), (40, 1281), (8, 6001)])
def test_band_nusselt_of_tall_cavities(nx, ny, storage, rounding):
    """Sums of a step by one warp and by a block, streams of one and of several rows."""
    assert_same(advance(nx, ny, storage, rounding, 0, runs=(6, 1, 530)), advance(nx, ny, storage, rounding, 2, runs=(6, 1, 530)))


def test_band_nusselt_short_ring_of_a_tall_cavity():
    assert_same(advance(40, 700, 0, 0, 0, cap=3), advance(40, 700, 0, 0, 2, cap=3))
