"""The level-set update as a launch per pass, the form for bands far beyond the one launch's
slots and for more level descriptors than a slot can name, against the persistent driver bit for
bit: a 2D and a 3D layer past the rule's line, and thousands of small cases (odd, padded and
periodic axes, frozen cases beside moving ones, iteration counts that skip passes, all lattices).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

PASSES = 2


def _layer(dims, periodic, block, lattice=None, seed=0, **over):
    D = len(dims)
    ax = [np.arange(n, dtype=np.float32) + 0.5 for n in dims]
    ph = np.random.default_rng(seed).uniform(0, 6, 2)
    x = ax[0].reshape((1,) * (D - 1) + (-1,))
    z = ax[D - 1].reshape((-1,) + (1,) * (D - 1))
    wave = 0.4 * np.sin(2 * np.pi * x / dims[0] + ph[0])
    if D == 3:
        wave = wave + 0.3 * np.sin(2 * np.pi * ax[1].reshape(1, -1, 1) / dims[1] + ph[1])
    wall = np.zeros((2 * D, D))
    wall[2 * D - 1, 0] = 0.02
    c = dict(lattice=lattice or ("D2Q9" if D == 2 else "D3Q19"), base=dims, n_levels=1, block=block, periodic=periodic,
             rho_phys=(1.0, 0.1), nu=(0.08, 0.3), sigma=2e-3, gravity=(0.0,) * (D - 1) + (-2e-5,),
             body_force=(1e-5,) + (0.0,) * (D - 1), wall_u=wall.reshape(-1),
             phi0=(z - 0.5 * dims[-1] - 0.3 - wave).astype(np.float32).reshape(-1))
    c.update(over)
    return c


def _state(cases, driver, steps, graphs):
    import torch

    from paper_2601_05936_gb300 import lsb
    g = lsb.Grid(cases, stream=torch.cuda.Stream())
    g.set_driver(driver)
    g.use_graphs(graphs)
    assert g.levelset_launch(0)["form"] == PASSES
    g.step(steps)
    g.sync()
    out = [g.get(f, k) for k in range(len(g.cases)) for f in ("phi", "uext", "rho", "u", "tag", "cutmask")]
    g.close()
    return out


def _both(cases, steps, graphs=True):
    for a, b in zip(_state(cases, 0, steps, graphs), _state(cases, 1, steps, False)):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("dims, block", [((163840, 40), (32, 8)), ((384, 384, 24), (32, 4, 4))])
def test_bands_far_beyond_the_slots(dims, block):
    _both(_layer(dims, (True,) * (len(dims) - 1) + (False,), block), steps=3)


@pytest.mark.parametrize("lattice", ["D2Q9", "D3Q19", "D3Q27"])
@pytest.mark.parametrize("over", [dict(), dict(n_ext=0), dict(n_ext=1, n_reinit=0), dict(n_ext=2, reinit_every=2, n_reinit=2)])
def test_more_descriptors_than_a_slot_can_name(lattice, over):
    D = 2 if lattice == "D2Q9" else 3
    sizes = [(16, 16), (5, 17), (12, 24)] if D == 2 else [(8, 4, 8), (5, 3, 9)]
    cases = [_layer(sizes[k % len(sizes)], tuple(a < D - 1 and (k >> a) & 1 == 0 for a in range(D)),
                    (8, 4) if D == 2 else (8, 2, 2), lattice, seed=k, ls_active=k % 5 != 0, **over)
             for k in range(4100)]
    _both(cases, steps=3, graphs="reinit_every" not in over)
