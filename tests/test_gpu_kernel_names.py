"""Kernel timing tells the forms of the level-set update apart, and has a name per form."""
import numpy as np
import pytest

from gpu_util import as_fp32_phi

pytestmark = pytest.mark.gpu


def _names(driver, moving=None):
    from paper_2601_05936_gb300 import lsb, workloads
    c = workloads.adjoint_window("D2Q9", seed=6055, n=(48, 32))
    if moving is not False:
        c.update(ls_active=True, n_ext=4, dtau_ext=0.5, reinit_every=1, n_reinit=1, dtau_reinit=0.3)
    g = lsb.Grid(as_fp32_phi(c))
    g.set_driver(driver)
    if moving is not None:
        g.record(2)
    g.step(2)
    g.profile(2)
    g.step(1) if moving is None else g.backward(np.ones((1, 8)), want_phi=True)
    names = set(g.profile_read())
    g.close()
    return names


def test_level_set_launches_are_told_apart():
    one, persistent = _names(0), _names(1)
    assert "k_levelset_fused" in one and not {"k_levelset_persistent", "k_classify_phase"} & one
    assert {"k_levelset_persistent", "k_classify_phase"} <= persistent and "k_levelset_fused" not in persistent


def test_reverse_sweep_names():
    frozen, moving = _names(0, False), _names(0, True)
    assert "k_adj_moments" in frozen and "k_lsa_levelset" not in frozen
    assert "k_lsa_levelset" in moving and "k_adj_moments" not in moving


def test_names_are_distinct():
    from paper_2601_05936_gb300 import lsb
    lib = lsb.load()
    names = [lib.lsb_kernel_name(k) for k in range(lib.lsb_kernel_count())]
    assert len(set(names)) == len(names)
