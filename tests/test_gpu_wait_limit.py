"""The wait limit in the launches that are the default: the one-launch level-set update where it
is a cooperative one, eager and captured, and the level-set launch of the reverse sweep.  With a
limit of zero each gives up at its first barrier, the next synchronising call reports
LSB_ETIMEOUT, and handles made afterwards give what they gave before.
"""
import numpy as np
import pytest

from gpu_util import as_fp32_phi

pytestmark = pytest.mark.gpu

ETIMEOUT = 5


def _wide_layer():
    """A band of 375 blocks: beyond a thread-block cluster, so the launch is cooperative."""
    nx, ny = 3000, 48
    X, Y = np.meshgrid(np.arange(nx) + 0.5, np.arange(ny) + 0.5)
    phi = Y - 24.3 - 0.4 * np.sin(2 * np.pi * X / nx)
    return dict(lattice="D2Q9", base=(nx, ny), block=(32, 8), periodic=(True, False), rho_phys=(1.0, 0.1),
                nu=(0.08, 0.3), sigma=2e-3, gravity=(0.0, -2e-5), phi0=phi.astype(np.float32).reshape(-1))


def _forward(graphs, limit=None):
    import torch

    from paper_2601_05936_gb300 import lsb
    g = lsb.Grid(_wide_layer(), stream=torch.cuda.Stream())
    g.use_graphs(graphs)
    g.step(2)
    g.sync()
    if limit is not None:
        g.set_wait_limit(limit)
    g.step(2)
    return g


@pytest.mark.parametrize("graphs", [False, True])
def test_forward_update_gives_up(graphs):
    from paper_2601_05936_gb300 import lsb
    ref = _forward(graphs).get("phi")
    g = _forward(graphs, 0)
    with pytest.raises(lsb.LsbError) as e:
        g.sync()
    assert e.value.status == ETIMEOUT
    g.step(1)  # the barrier's words are clear again: the next launch ends as well
    with pytest.raises(lsb.LsbError) as e:
        g.sync()
    assert e.value.status == ETIMEOUT
    g.close()
    ok = _forward(graphs)
    assert np.array_equal(ok.get("phi"), ref)
    ok.close()


def _window(levels, limit=None):
    from paper_2601_05936_gb300 import lsb, workloads
    kw = dict(n=(48, 32), seed=6055) if levels == 1 else dict(n=(48, 24), seed=6158, levels=2, block=(8, 8))
    case = workloads.adjoint_window("D2Q9", **kw)
    case.update(ls_active=True, n_ext=4, dtau_ext=0.5, reinit_every=1, n_reinit=1, dtau_reinit=0.3)
    g = lsb.Grid(as_fp32_phi(case))
    g.step(2)
    g.record(2)
    g.step(3)
    g.sync()
    if limit is not None:
        g.set_wait_limit(limit)
    return g


@pytest.mark.parametrize("levels", [1, 2])
def test_reverse_sweep_gives_up(levels):
    from paper_2601_05936_gb300 import lsb
    w = np.random.default_rng(7).standard_normal((1, 8))
    ref, _ = _window(levels).backward(w, want_phi=True)
    g = _window(levels, 0)
    with pytest.raises(lsb.LsbError) as e:
        g.backward(w, want_phi=True)
    assert e.value.status == ETIMEOUT
    g.close()
    dp, _ = _window(levels).backward(w, want_phi=True)
    # the atomics' order is the only difference: FP32 rounding times the terms of a sum
    assert np.allclose(dp, ref, rtol=1e-4, atol=1e-12)
