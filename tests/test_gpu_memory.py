"""Device memory of a handle, per finest cell of a single-level 3D grid (D3Q19, FP32).

Two population buffers 152 bytes; phi, two stage arrays, S(phi0) and frozen flags 17; u~ 12 and its two
sweep buffers 32; cut mask and link base 8; interface moments 48, normal and curvature 16; links 34;
interface and flip lists 4; tag 1: 324.  A layout that needs more than 333 would no longer hold every grid
that the separate plan arrays and unpadded records of earlier layouts held.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _used():
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    return -free


def _box(n):
    z = (np.arange(n, dtype=np.float32) + 0.5).reshape(-1, 1, 1)
    return dict(lattice="D3Q19", base=(n, n, n), block=(32, 4, 4), periodic=(True, True, False), rho_phys=(1.0, 0.1),
                nu=(0.1, 0.1), sigma=0.0, phi0=np.broadcast_to(z - 0.5 * n - 0.3, (n, n, n)).reshape(-1))


def test_bytes_per_finest_cell():
    from paper_2601_05936_gb300 import lsb
    n = 256
    lsb.Grid(_box(32)).close()  # context, modules
    before = _used()
    g = lsb.Grid(_box(n))
    g.step(2)
    g.sync()
    used = _used() - before
    g.close()
    # allocations are rounded to 2 MiB: some 40 of them beside the cells' own bytes
    assert used <= 333 * n ** 3 + 96 * 2 ** 20, used / n ** 3
