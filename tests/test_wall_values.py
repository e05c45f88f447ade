"""Wall profiles that an adiabatic wall does not use: whatever they hold, the state is that
of the one-step kernel (its wall value is the node's own opposite and nothing else)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

MARCH, BAND = 4, 5


def run(nx, ny, storage, kernel, walls, bad, expect=None):
    from paper_1601_04633_gb300 import dmrt as D

    rng = np.random.default_rng(nx + ny)
    p = D.make_params(nx, ny, 1e4, 0.01, storage=storage, kernel=kernel, nu_capacity=64, left_wall=walls[0],
                      right_wall=walls[1])
    sim = D.Cavity2D(p, theta0=0.3 * rng.standard_normal((ny, nx)))
    profile = np.full(ny, bad)
    D.dmrt_set_wall_profiles(sim.h, hot=profile if walls[0] else None, cold=profile if walls[1] else None)
    if expect:
        assert sim.run_launch(9)["kernel"] == expect
    sim.step(9)
    sim.check()
    out = [sim.get_state(), sim.nusselt(64)[2]]
    sim.close()
    assert np.isfinite(out[0]).all()
    return out


@pytest.mark.parametrize("nx,ny,kernel", [(449, 891, MARCH), (131, 160, BAND), (64, 64, BAND)])
@pytest.mark.parametrize("walls", [(1, 0), (0, 1), (1, 1)])
@pytest.mark.parametrize("storage,bad", [(0, np.nan), (3, np.inf), (4, np.nan), (1, 1e300)])
def test_an_adiabatic_wall_ignores_its_profile(nx, ny, kernel, walls, storage, bad):
    for a, b in zip(run(nx, ny, storage, 0, walls, bad, kernel), run(nx, ny, storage, 2, walls, bad)):
        np.testing.assert_array_equal(a, b)
