"""Runs that only the march kernel takes (cavities too wide or too large for the band
kernel): chains of three-step launches, graphs of them, their Nusselt hand-over and
every remainder, against the one-step TMA kernel, bit for bit."""
import os
import subprocess
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

pytestmark = pytest.mark.gpu

MARCH = 4
# Launches from either buffer; 200 and 400: one and two graphs of 192 steps, remainders of
# 8 = 3 + 2 + 2 + 1 steps (3 + 3 + 1 + 1 in 16-bit storage) and 16.
RUNS = (3, 200, 1, 400, 4, 2, 5, 7, 6, 1)
MODES = [(0, 0), (1, 0), (1, 1), (2, 0), (2, 1), (3, 0), (3, 1), (4, 0), (4, 1)]
# Whole strips (60 columns in float32, 56 in 16-bit storage), one column more or less, several
# chunks, few rows, and more than 1024 rows (Nusselt sums of several rows per partial);
# 16-bit storage marches from 400000 nodes on up to 900 columns, above 1600 from a million.
SIZES = [(1080, 43), (1081, 171), (1064, 181), (1063, 90), (777, 701), (241, 1501)]
SIZES16 = [(448, 900), (447, 901), (449, 891), (241, 1701), (1065, 951), (5001, 201)]
CASES = [(nx, ny, st, rd) for st, rd in MODES for nx, ny in (SIZES16 if st else SIZES)]


def advance(nx, ny, storage, rounding, kernel, walls=(0, 0), cap=4096, runs=RUNS):
    from paper_1601_04633_gb300 import dmrt as D

    p = D.make_params(nx, ny, min(1e4, 0.01 * (12 * ny) ** 2), 0.01, storage=storage, rounding=rounding, kernel=kernel,
                      nu_capacity=cap, left_wall=walls[0], right_wall=walls[1], theta_ref=0.1)
    rng = np.random.default_rng(nx * 10007 + ny)
    sim = D.Cavity2D(p, theta0=0.3 * rng.standard_normal((ny, nx)),
                     theta_hot_profile=0.5 + 0.01 * rng.standard_normal(ny))
    if kernel == 0:
        assert all(sim.run_launch(n)["kernel"] == MARCH for n in (200, 400))
    out = []
    for n in runs:
        sim.step(n)
        mean, rows, _ = sim.nusselt(1)
        out += [np.array(mean), rows]
    sim.check()
    out += [sim.get_state(), sim.nusselt(cap)[2]] + [t.cpu().numpy() for t in sim.fields()]
    sim.close()
    return out


def assert_same(a, b):
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("nx,ny,storage,rounding", CASES)
def test_march_chain_equals_single_steps(nx, ny, storage, rounding):
    assert_same(advance(nx, ny, storage, rounding, 0), advance(nx, ny, storage, rounding, 2))


@pytest.mark.parametrize("nx,ny,storage,rounding", [(1030, 511, 0, 0), (1030, 512, 0, 0), (300, 1023, 0, 0), (167, 4100, 0, 0),
                                                    (167, 4100, 1, 1), (420, 1023, 3, 1)])
def test_march_chain_tall_cavities(nx, ny, storage, rounding):
    """Nusselt sums by one, two, three and eight blocks."""
    assert_same(advance(nx, ny, storage, rounding, 0), advance(nx, ny, storage, rounding, 2))


@pytest.mark.parametrize("storage,rounding", [(0, 0), (3, 1)])
def test_march_chain_of_a_batch_with_a_tall_member(storage, rounding):
    from paper_1601_04633_gb300 import dmrt as D
    from paper_1601_04633_gb300 import inputs

    cavs = [inputs.Cavity(nx, ny, min(1e4, 0.01 * (12 * ny) ** 2), 0.01, noise_amp=1e-2, seed=k)
            for k, (nx, ny) in enumerate(((60, 2100), (130, 19), (57, 300), (8, 8)))]
    b = D.Batch.from_inputs(cavs, nu_capacity=512, storage=storage, rounding=rounding)
    assert b.run_launch(30)["kernel"] == MARCH
    for n in (30, 1, 4, 5, 7, 64):
        b.step(n)
    b.check()
    for m, c in zip(b.members, cavs):
        ref = D.Cavity2D.from_inputs(c, nu_capacity=512, storage=storage, rounding=rounding, kernel=2)
        ref.step(111)
        got, want = m.nusselt(512), ref.nusselt(512)
        assert_same([m.get_state(), got[1], got[2]], [ref.get_state(), want[1], want[2]])
        ref.close()
    b.close()


@pytest.mark.parametrize("count,storage,rounding", [(80, 0, 0), (81, 0, 0), (81, 3, 1), (163, 3, 0)])
def test_march_chain_of_several_groups_of_a_batch(count, storage, rounding):
    """Groups of up to 80 cavities, single steps and short runs in between, every member."""
    from paper_1601_04633_gb300 import dmrt as D
    from paper_1601_04633_gb300 import inputs

    cavs = [inputs.Cavity(8 + k % 61, 8 + k % 23, 1e3, 0.01, noise_amp=1e-2, seed=k) for k in range(count)]
    b = D.Batch.from_inputs(cavs, nu_capacity=64, storage=storage, rounding=rounding)
    for n in (1, 3, 2, 4, 1, 5, 9, 8):
        b.step(n)
    b.check()
    for m, c in zip(b.members, cavs):
        ref = D.Cavity2D.from_inputs(c, nu_capacity=64, storage=storage, rounding=rounding, kernel=2)
        ref.step(33)
        assert_same([m.get_state(), m.nusselt(64)[2]], [ref.get_state(), ref.nusselt(64)[2]])
        ref.close()
    b.close()


@pytest.mark.parametrize("walls", [(1, 0), (0, 1), (1, 1)])
@pytest.mark.parametrize("storage", [0, 1, 3, 4])
def test_march_chain_wall_kinds(walls, storage):
    nx, ny = (449, 891) if storage else (1081, 171)
    assert_same(advance(nx, ny, storage, 2, 0, walls), advance(nx, ny, storage, 2, 2, walls))


@pytest.mark.parametrize("cap", [1, 2, 3, 5])
def test_march_chain_short_nusselt_ring(cap):
    assert_same(advance(1081, 171, 0, 0, 0, cap=cap), advance(1081, 171, 0, 0, 2, cap=cap))


def test_march_chain_bounds_checked_build():
    code = ("import sys; sys.path.insert(0, %r); from tests.test_march_chain import advance;"
            "[advance(nx, ny, s, 2, 0) for nx, ny in ((449, 891), (241, 1701)) for s in range(5)]" % ROOT)
    subprocess.run([sys.executable, "-c", code], check=True, cwd=ROOT,
                   env=dict(os.environ, DMRT_LIBRARY="bounds_check"))
