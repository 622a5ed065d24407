"""The one-launch level-set update keeps to the band it has, where no regrid plans it anew.

Two vertical interfaces between walls that move against each other: on one level nothing regrids,
and the band grows from 96 blocks, a cluster's, beyond the 128 that a cluster has slots for.  The launch has to
hold the grown band in its slots again after every synchronising call, and within a stretch of
steps without one; a band that vanishes takes the launch with it.  The state is the persistent
driver's, bit for bit, whatever shape the steps ran with.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CLUSTER, GRID = 0, 1


def _sheared(nx=512, ny=96, U=0.08):
    X = np.broadcast_to(np.arange(nx) + 0.5, (ny, nx))
    phi = np.abs(X - nx / 2) - nx / 4
    wall = np.zeros((4, 2))
    wall[2, 0], wall[3, 0] = -U, U
    return dict(lattice="D2Q9", base=(nx, ny), block=(32, 8), periodic=(True, False), rho_phys=(1.0, 1.0), nu=(0.3, 0.3),
                sigma=0.0, wall_u=wall.reshape(-1), phi0=phi.astype(np.float32).reshape(-1))


def _grid(case, driver=0, graphs=True):
    import torch

    from paper_2601_05936_gb300 import lsb
    g = lsb.Grid(case, stream=torch.cuda.Stream())
    g.set_driver(driver)
    g.use_graphs(graphs)
    return g


def _same(a, b):
    for f in ("phi", "uext", "rho", "u", "tag", "cutmask"):
        assert np.array_equal(a.get(f), b.get(f)), f


@pytest.mark.parametrize("graphs", [False, True])
def test_followed_after_synchronising_calls(graphs):
    g = _grid(_sheared(), graphs=graphs)
    band0, shape0 = g.work_counts(0)["band"], g.levelset_launch(0)
    for _ in range(20):
        g.step(100)
        g.sync()
        g.step(1)  # plans before its launches, for the band that the synchronising call saw
        assert g.levelset_launch(0)["cells"] >= g.work_counts(0)["band"]
    assert g.work_counts(0)["band"] > shape0["cells"] >= band0 and g.levelset_launch(0) != shape0
    ref = _grid(_sheared(), driver=1, graphs=graphs)
    ref.step(2020)
    _same(g, ref)
    g.close()
    ref.close()


def test_followed_within_one_call():
    """Eager steps: the launches queue ahead of the GPU by a few hundred steps at most."""
    g, ref = _grid(_sheared(), graphs=False), _grid(_sheared(), driver=1)
    shape0 = g.levelset_launch(0)
    g.step(2020)
    assert g.levelset_launch(0) != shape0
    ref.step(2020)
    _same(g, ref)
    g.close()
    ref.close()


def test_band_that_vanishes():
    """A drop of three cells that the reinitialised transport loses, then a field without interface."""
    n = 96
    X, Y = np.meshgrid(np.arange(n) + 0.5, np.arange(n) + 0.5)
    case = _sheared()
    case.update(base=(n, n), phi0=(1.2 - np.hypot(X - 48.2, Y - 50.3)).astype(np.float32).reshape(-1))
    g, ref = _grid(case), _grid(case, driver=1)
    for _ in range(6):
        g.step(200)
        g.sync()
    g.step(2)
    ref.step(1202)
    _same(g, ref)
    if g.work_counts(0)["band"] == 0:
        assert g.levelset_launch(0)["ctas"] == 1
    g.close()
    ref.close()


def test_stepping_inside_a_capture():
    """Steps captured by the caller keep the plan they were captured with: no copy, query or new
    plan meanwhile.  Replayed while the band outgrows the slots of its cluster, the cells beyond them
    take the per-cell functions beside a pass without a barrier before it."""
    import torch

    from paper_2601_05936_gb300 import lsb
    s = torch.cuda.Stream()
    g = lsb.Grid(_sheared(), stream=s)
    ref = lsb.Grid(_sheared(), stream=torch.cuda.Stream())
    ref.set_driver(1)
    g.step(2)
    g.sync()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        g.step(80)  # beyond the steps after which the band is looked at
    for _ in range(26):
        graph.replay()
    torch.cuda.synchronize()
    shape = g.levelset_launch(0)
    assert shape["form"] == CLUSTER and g.work_counts(0)["band"] > shape["cells"]
    ref.step(2082)
    _same(g, ref)
    g.close()
    ref.close()


@pytest.mark.parametrize("dims, block, form, slots", [
    ((8, 8), (8, 4), CLUSTER, 1), ((256, 48), (32, 8), CLUSTER, 1), ((1000, 48), (32, 8), CLUSTER, 2),
    ((3000, 48), (32, 8), GRID, 1), ((64, 64, 24), (16, 8, 4), GRID, 1), ((256, 256, 32), (32, 4, 4), GRID, 5)])
def test_shapes_that_the_launch_tests_cover(dims, block, form, slots):
    """The sizes of test_gpu_levelset_launch.py reach the forms they stand for; the last one has more
    band cells than the grid holds."""
    from test_gpu_levelset_launch import _layers
    g = _grid(_layers(dims, (True,) * (len(dims) - 1) + (False,), block))
    shape, band = g.levelset_launch(0), g.work_counts(0)["band"]
    assert shape["form"] == form and shape["cells"] == slots * shape["ctas"] * shape["threads"], (shape, band)
    assert (band > shape["cells"]) == (dims == (256, 256, 32)), (shape, band)
    g.close()
