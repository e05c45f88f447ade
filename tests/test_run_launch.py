"""dmrt_get_run_launch / dmrt_batch_get_run_launch: the kernel that takes a run of steps
under AUTO, so that a comparison of AUTO with a named kernel compares two kernels."""
import pytest

pytestmark = pytest.mark.gpu

DIRECT, TMA, CLUSTER, MARCH, BAND = 1, 2, 3, 4, 5


@pytest.fixture(scope="module")
def D():
    import __graft_entry__

    __graft_entry__.build()
    from paper_1601_04633_gb300 import dmrt

    return dmrt


def plan(D, nx, ny, n, storage=0, **kw):
    sim = D.Cavity2D(D.make_params(nx, ny, 1e4, 0.01, storage=storage, nu_capacity=16, **kw))
    r = sim.run_launch(n)
    sim.close()
    return r


@pytest.mark.parametrize("nx,ny,storage,n,kernel,cluster,launches", [
    # Sizes from which a storage marches; two-step launches in float32 only; float16 and
    # bfloat16 (and THETA32 below 1200000 nodes, mixed below 600000) runs of six steps or more.
    (1100, 40, 0, 4, MARCH, 0, 3), (1000, 39, 0, 10, BAND, 0, 2), (1100, 36, 0, 10, TMA, 0, 11),
    (800, 499, 3, 30, TMA, 0, 31), (800, 500, 3, 30, MARCH, 0, 11), (800, 500, 1, 6, MARCH, 0, 3), (800, 499, 1, 6, TMA, 0, 7),
    (1600, 343, 4, 30, TMA, 0, 31), (1600, 344, 4, 30, MARCH, 0, 11), (1601, 344, 4, 30, TMA, 0, 31), (901, 610, 3, 30, TMA, 0, 31), (900, 610, 4, 30, MARCH, 0, 11), (1700, 353, 3, 30, MARCH, 0, 11), (1700, 352, 3, 30, TMA, 0, 31),
    (2000, 499, 1, 30, TMA, 0, 31), (2000, 500, 1, 30, MARCH, 0, 11),
    (1100, 545, 3, 4, TMA, 0, 5), (1100, 546, 3, 4, MARCH, 0, 4), (1100, 910, 1, 5, TMA, 0, 6), (1100, 910, 2, 8, MARCH, 0, 2 + 1 + 2 + 1),
    (1100, 1090, 4, 5, TMA, 0, 6), (1100, 1091, 4, 5, MARCH, 0, 1 + 1 + 2 + 1),
    (300, 300, 4, 5, TMA, 0, 6), (300, 300, 0, 5, MARCH, 0, 5), (159, 9000, 0, 30, DIRECT, 0, 31),
    (32, 32, 0, 100, CLUSTER, 1, 2),          # and the Nusselt sum
    (64, 64, 0, 5, CLUSTER, 1, 2),
    # One-row blocks: the cluster kernel up to 352 columns, and from 513 on while it holds them.
    (300, 16, 0, 50, CLUSTER, 1, 2), (352, 10, 0, 50, CLUSTER, 1, 2), (353, 10, 0, 50, BAND, 1, 2),
    (512, 4, 0, 50, BAND, 1, 2), (513, 16, 0, 50, CLUSTER, 1, 2), (640, 3, 0, 50, CLUSTER, 1, 2), (1000, 2, 0, 50, BAND, 0, 2),
    # Wide and flat in 16-bit storage: a launch per step.
    (751, 106, 1, 50, TMA, 0, 51), (751, 107, 1, 50, BAND, 0, 2), (750, 8, 3, 50, BAND, 0, 2), (1024, 60, 0, 50, BAND, 0, 2),
    (64, 64, 0, 2000, BAND, 1, 8),            # four launches and their sums
    (64, 64, 3, 2000, BAND, 1, 8),
    (256, 256, 0, 515, BAND, 0, 4),
    (512, 512, 4, 100, BAND, 0, 2),
    (1100, 900, 0, 5 * 192 + 30, MARCH, 0, 331),
    (2048, 2048, 3, 9, MARCH, 0, 4),
    (2048, 2048, 0, 4, MARCH, 0, 3),          # two launches of two steps
    (2048, 2048, 0, 2, TMA, 0, 3),
])
def test_the_kernel_of_a_run(D, nx, ny, storage, n, kernel, cluster, launches):
    r = plan(D, nx, ny, n, storage)
    assert (r["kernel"], r["cluster"], r["launches"]) == (kernel, cluster, launches)
    assert 0 <= n - r["steps"] < 3 and r["grid"] > 0 and r["block"] > 0  # (a remainder goes in single steps)
    assert r["graph_steps"] == (192 if kernel == MARCH and n >= 192 else 0)


def test_a_named_kernel_or_tile_takes_one_step_per_launch(D):
    for kw in ({"kernel": TMA}, {"kernel": TMA, "tma_rows": 2, "tma_npt": 2, "tma_stages": 2}):
        r = plan(D, 256, 256, 100, **kw)
        assert (r["kernel"], r["steps_per_launch"], r["launches"], r["graph_steps"]) == (TMA, 1, 101, 64)
    assert plan(D, 64, 64, 100, kernel=CLUSTER)["kernel"] == CLUSTER


def test_batch_runs(D):
    from paper_1601_04633_gb300 import inputs

    cavs = [inputs.Cavity(100 + 30 * k, 150, 1e4, 0.01) for k in range(5)]
    for opts, n, want in ((None, 256, (MARCH, 3, 86 + 1)), (None, 5, (MARCH, 2, 2 + 1 + 1 + 1)), (None, 2, (TMA, 1, 3)),
                          ({"tma_npt": 2, "tma_rows": 2, "tma_stages": 2}, 100, (TMA, 1, 101)),
                          ({"tma_npt": 2, "tma_rows": 2, "tma_stages": 2, "steps_per_launch": 8}, 100, (TMA, 8, 12 + 4 + 1))):
        b = D.Batch.from_inputs(cavs, opts=opts, nu_capacity=16)
        r = b.run_launch(n)
        assert (r["kernel"], r["steps_per_launch"], r["launches"]) == want
        b.close()
    # Mixed storage leaves a remainder to single steps; more than 80 cavities: groups, each with its launches.
    for count, storage, n, launches in ((5, 3, 5, 1 + 1 + 2 + 1), (81, 0, 6, 2 * (2 + 1))):
        b = D.Batch.from_inputs([inputs.Cavity(20, 20, 1e3, 0.01)] * count, nu_capacity=16, storage=storage)
        r = b.run_launch(n)
        assert (r["kernel"], r["steps_per_launch"], r["launches"]) == (MARCH, 3, launches)
        b.close()
