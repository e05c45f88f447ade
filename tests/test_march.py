"""The march kernel (several steps per launch, AUTO's choice for runs of steps of
larger cavities) against the one-step TMA kernel: a launch gives the bits of
its single steps, in every storage mode and rounding, at the edges of its strips
(60 columns in float32, 56 in 16-bit storage), of its row chunks, and for every
remainder of a run after launches of three and two steps."""
import os
import subprocess
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

pytestmark = pytest.mark.gpu

RUNS = (1, 2, 3, 4, 5, 7, 200, 1)  # 200: past a graph of 64 launches
MODES = [(0, 0), (1, 0), (1, 1), (2, 0), (2, 1), (3, 0), (3, 1), (4, 0), (4, 1)]
SIZES = [(60 * 4, 170), (60 * 4 + 1, 171), (56 * 4, 181), (56 * 4 - 1, 180), (160, 251), (181, 667), (5000, 9), (383, 389)]


def advance(nx, ny, storage, rounding, kernel, walls=(0, 0), cap=4096):
    from paper_1601_04633_gb300 import dmrt as D

    p = D.make_params(nx, ny, 1e4, 0.01, storage=storage, rounding=rounding, kernel=kernel, nu_capacity=cap,
                      left_wall=walls[0], right_wall=walls[1], theta_ref=0.1)
    rng = np.random.default_rng(nx * 10007 + ny)
    sim = D.Cavity2D(p, theta0=0.3 * rng.standard_normal((ny, nx)),
                     theta_hot_profile=0.5 + 0.01 * rng.standard_normal(ny))
    for n in RUNS:
        sim.step(n)
    sim.check()
    mean, rows, series = sim.nusselt(cap)
    out = [sim.get_state(), rows, series, np.array(mean)] + [t.cpu().numpy() for t in sim.fields()]
    sim.close()
    return out


def test_march_members_stay_in_phase():
    """A batch takes members that were stepped alone by an even number of steps."""
    from paper_1601_04633_gb300 import dmrt as D
    from paper_1601_04633_gb300 import inputs

    cavs = [inputs.Cavity(230, 200, 1e4, 0.01, seed=s) for s in (1, 2)]
    for n in (2, 4, 6, 8, 10, 14):
        b = D.Batch.from_inputs(cavs, nu_capacity=64)
        b.members[0].step(n)
        b.step(3)
        b.members[1].step(n)
        b.check()
        states = [m.get_state() for m in b.members]
        b.close()
        for c, got in zip(cavs, states):
            sim = D.Cavity2D.from_inputs(c, kernel=D.DMRT_KERNEL_TMA, nu_capacity=64)
            sim.step(n + 3)
            np.testing.assert_array_equal(sim.get_state(), got)
            sim.close()


@pytest.mark.parametrize("storage,rounding", [(0, 0), (3, 0), (3, 1)])
@pytest.mark.parametrize("count", [1, 3, 70])
def test_march_batch_equals_members_alone(count, storage, rounding):
    """Batches stepped by march launches (no tile asked for), one and two groups of
    cavities, with single steps and members stepped alone in between."""
    from paper_1601_04633_gb300 import dmrt as D
    from paper_1601_04633_gb300 import inputs

    rng = np.random.default_rng(count)
    cavs = []
    for k in range(count):
        nx, ny = int(rng.integers(8, 150) if count > 3 else rng.integers(100, 400)), int(rng.integers(20, 150))
        cavs.append(inputs.Cavity(nx, ny, min(1e4, 0.01 * (12 * ny) ** 2), 0.01, noise_amp=1e-2, seed=k))
    b = D.Batch.from_inputs(cavs, nu_capacity=512, storage=storage, rounding=rounding)
    for n in RUNS[:6] + (64, 8, 1):
        b.step(n)
    b.members[0].step(4)
    b.step(3)
    b.check()
    total = sum(RUNS[:6]) + 64 + 8 + 1 + 3
    for i in range(0, count, 9 if count > 3 else 1):
        ref = D.Cavity2D.from_inputs(cavs[i], nu_capacity=512, storage=storage, rounding=rounding, kernel=2)
        ref.step(total + (4 if i == 0 else 0))
        got, want = b.members[i].nusselt(512), ref.nusselt(512)
        np.testing.assert_array_equal(b.members[i].get_state(), ref.get_state())
        np.testing.assert_array_equal(got[2], want[2])
        np.testing.assert_array_equal(got[1], want[1])
        ref.close()
    b.close()


def assert_same(a, b):
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("storage,rounding", MODES)
@pytest.mark.parametrize("nx,ny", SIZES)
def test_march_equals_single_steps(nx, ny, storage, rounding):
    assert nx * ny >= 40000 and nx >= 160  # the sizes that AUTO marches
    assert_same(advance(nx, ny, storage, rounding, 0), advance(nx, ny, storage, rounding, 2))


@pytest.mark.parametrize("walls", [(1, 0), (0, 1), (1, 1)])
@pytest.mark.parametrize("storage", [0, 3, 4])
def test_march_wall_kinds(walls, storage):
    assert_same(advance(243, 170, storage, 2, 0, walls), advance(243, 170, storage, 2, 2, walls))


@pytest.mark.parametrize("cap", [1, 2, 5])
def test_march_short_nusselt_ring(cap):
    assert_same(advance(243, 170, 0, 0, 0, cap=cap), advance(243, 170, 0, 0, 2, cap=cap))


def test_march_bounds_checked_build():
    code = ("import sys; sys.path.insert(0, %r); from tests.test_march import advance;"
            "[advance(nx, ny, s, 2, 0) for nx, ny in ((241, 171), (160, 251), (223, 180)) for s in range(5)]" % ROOT)
    subprocess.run([sys.executable, "-c", code], check=True, cwd=ROOT,
                   env=dict(os.environ, DMRT_LIBRARY="bounds_check"))
