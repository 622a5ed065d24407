"""The one-launch level-set update (driver 0) against the per-pass lookups of the persistent
driver (driver 1), bit for bit, at the sizes where the launch changes shape: one block, a
cluster of every size, two cells per thread of the largest cluster, a cooperative grid, and
bands with more cells than the slots in shared memory; short, odd and periodic axes; the
iteration counts that skip passes; frozen cases beside moving ones; more level descriptors
than the table in shared memory; and two handles on streams of their own at a time."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _layers(dims, periodic, block, h=None, seed=0, **over):
    """Liquid below gas along the last axis with a wavy interface, a moving lid and gravity."""
    D = len(dims)
    rng = np.random.default_rng(seed)
    X = np.meshgrid(*[np.arange(n) + 0.5 for n in dims[::-1]], indexing="ij")[::-1]
    h = 0.5 * dims[-1] + 0.3 if h is None else h
    wave = 0.4 * np.sin(2 * np.pi * X[0] / dims[0] + rng.uniform(0, 6))
    if D == 3:
        wave = wave + 0.3 * np.sin(2 * np.pi * X[1] / dims[1] + rng.uniform(0, 6))
    wall = np.zeros((2 * D, D))
    wall[2 * D - 1, 0] = 0.02
    c = dict(lattice="D2Q9" if D == 2 else "D3Q19", base=dims, n_levels=1, block=block, periodic=periodic,
             rho_phys=(1.0, 0.1), nu=(0.08, 0.3), sigma=2e-3, gravity=(0.0,) * (D - 1) + (-2e-5,),
             body_force=(1e-5,) + (0.0,) * (D - 1), wall_u=wall.reshape(-1),
             phi0=(X[D - 1] - h - wave).astype(np.float32).reshape(-1))
    c.update(over)
    return c


def _state(g):
    out = []
    for k, c in enumerate(g.cases):
        out += [g.get(f, k) for f in ("phi", "uext", "rho", "u", "tag", "cutmask")]
    return out


def _run(cases, driver, steps):
    import torch

    from paper_2601_05936_gb300 import lsb
    g = lsb.Grid(cases, stream=torch.cuda.Stream())
    g.set_driver(driver)
    g.step(steps)
    g.sync()
    out = _state(g)
    g.close()
    return out


def _both(cases, steps=4):
    for a, b in zip(_run(cases, 0, steps), _run(cases, 1, steps)):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("dims, block", [
    ((8, 8), (8, 4)),            # one column of blocks, axes shorter than the blocks' reach
    ((5, 24), (8, 8)),           # padded and odd, periodic axis of 5
    ((32, 40), (32, 8)),         # a cluster of a few CTAs
    ((256, 48), (32, 8)),        # the full cluster, one cell per thread
    ((1000, 48), (32, 8)),       # two cells per thread
    ((3000, 48), (32, 8)),       # the cooperative grid
])
@pytest.mark.parametrize("periodic", [True, False])
def test_launch_shapes_2d(dims, block, periodic):
    _both(_layers(dims, (periodic, False), block))


@pytest.mark.parametrize("dims, block", [
    ((16, 3, 24), (16, 2, 4)),   # an axis of three cells
    ((33, 17, 24), (32, 4, 4)),  # odd, padded
    ((64, 64, 24), (16, 8, 4)),
    ((256, 256, 32), (32, 4, 4)),  # more band cells than slots
])
@pytest.mark.parametrize("periodic", [(True, True, False), (False, False, False)])
def test_launch_shapes_3d(dims, block, periodic):
    _both(_layers(dims, periodic, block), steps=3)


@pytest.mark.parametrize("over", [dict(n_ext=0), dict(n_ext=1), dict(n_ext=2, reinit_every=0),
                                  dict(reinit_every=2, n_reinit=2), dict(n_reinit=0), dict(n_reinit=3)])
def test_iteration_counts(over):
    _both(_layers((48, 40), (True, False), (32, 8), **over), steps=5)


def test_frozen_beside_moving_and_many_descriptors():
    """200 small cases (more descriptors than the shared table), every third with its level set frozen."""
    cases = [_layers((32, 24 + 2 * (k % 5)), (k % 2 == 0, False), (32, 8), seed=k, ls_active=k % 3 != 0)
             for k in range(200)]
    _both(cases, steps=3)


def test_no_interface():
    _both(_layers((64, 32), (True, False), (32, 8), phi0=-np.ones(64 * 32, np.float32)))


def test_two_handles_at_a_time():
    """Two handles whose level-set launches both want every SM, stepped from two threads."""
    import torch

    from paper_2601_05936_gb300 import lsb
    cases = [_layers((128, 128, 48), (True, True, False), (32, 4, 4), seed=s) for s in (1, 2)]
    ref = [_run(c, 0, 12) for c in cases]
    grids = [lsb.Grid(c, stream=torch.cuda.Stream()) for c in cases]

    def go(g):
        for _ in range(12):
            g.step(1)
        g.sync()

    ts = [threading.Thread(target=go, args=(g,)) for g in grids]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for g, r in zip(grids, ref):
        for a, b in zip(_state(g), r):
            assert np.array_equal(a, b)
        g.close()
