"""The cut links' part of the frozen window's reverse sweep over many cases in one handle.

With a frozen level set one thread takes one cut link; the links of all cases lie in one list, so
a warp can hold links of several cases, and beyond 64 cases the parameter partials go to global
memory instead of shared.  Every case of an uneven ensemble has to give what it gives alone: the
links' macro adjoints meet in atomics, whose order is the only difference, so lambda differs by FP32
rounding (6e-8) times the few dozen terms of a cell and the steps of the window, and the FP64
parameter sums by that of lambda: 1e-5 relative, 1e-4 for dJ/dphi with its 1/(phi_x - phi_y)^2.
"""
import numpy as np
import pytest

from gpu_util import as_fp32_phi, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,sizes,ncase", [("D2Q9", ((32, 24), (45, 23), (33, 40)), 3),
                                                 ("D2Q9", ((32, 24), (19, 21), (27, 18)), 66),
                                                 ("D3Q19", ((24, 13, 17), (32, 16, 20)), 2)])
def test_links_of_many_cases(lattice, sizes, ncase):
    from paper_2601_05936_gb300 import lsb, workloads
    D, steps = len(sizes[0]), 4
    cases = [as_fp32_phi(workloads.adjoint_window(lattice, n=sizes[i % len(sizes)], seed=6100 + i % (2 * len(sizes))))
             for i in range(ncase)]
    a = np.random.default_rng(5).standard_normal((ncase, 4 + 2 * D))

    def sweep(cs, w):
        g = lsb.Grid(cs)
        g.step(3)
        g.record(steps)
        g.step(steps)
        dp, dphi = g.backward(w, want_phi=True)
        g.close()
        return np.asarray(dp), [np.asarray(p, dtype=np.float64).reshape(-1) for p in dphi]

    dp, dphi = sweep(cases, a)
    for k in sorted({0, 1, ncase // 2, ncase - 1}):
        one, phi1 = sweep([cases[k]], a[k:k + 1])
        assert np.abs(dp[k] - one[0]).max() <= 1e-5 * np.abs(one[0]).max(), (k, dp[k], one[0])
        assert (np.abs(dp[k] - one[0]) <= 1e-4 * np.abs(one[0]) + 1e-9).all(), (k, dp[k], one[0])
        assert rel_l2(dphi[k], phi1[0]) < 1e-4, k
