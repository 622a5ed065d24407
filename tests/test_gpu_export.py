"""Fields exported to device memory: written by the export kernel itself, or through staging.

A float-aligned destination inside one allocation of the current device is written directly; an odd
address takes the staged copy.  All of them hold the bytes that the export to the host gives, and
nothing past the field is touched.
"""
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,n,block,storage,levels", [
    ("D2Q9", (33, 25), (32, 8), "fp32", 1), ("D2Q9", (32, 40), (16, 16), "fp16s", 2),
    ("D3Q19", (19, 23, 21), (32, 4, 4), "fp32", 1), ("D3Q27", (16, 16, 32), (16, 4, 4), "fp32", 1)])
def test_device_export_matches_host(lattice, n, block, storage, levels):
    from paper_2601_05936_gb300 import lsb, workloads
    if lattice == "D3Q27":
        case = workloads.paper_box_3d("I", d=8, block=block, nu_floor=0.1, lattice=lattice)
    else:
        case = workloads.adjoint_window(lattice, n=n, levels=levels, block=block)
    case["storage"] = storage
    g = lsb.Grid(case)
    g.step(3)
    for level in range(levels):
        for field in ("rho", "u", "f"):
            host = g.get(field, level=level)
            nb = host.nbytes
            for off in (0, 4, 12, 1, 6):  # 1 and 6: not float-aligned
                buf = torch.full((nb + 64,), 0xA5, dtype=torch.uint8, device="cuda")
                torch.cuda.synchronize()
                g.get_device(field, buf.data_ptr() + off, nb, level=level)
                got = buf.cpu().numpy()
                assert (got[off:off + nb] == host.reshape(-1).view(np.uint8)).all(), (field, level, off)
                assert (got[:off] == 0xA5).all() and (got[off + nb:] == 0xA5).all(), (field, level, off)
            small = torch.empty(nb, dtype=torch.uint8, device="cuda")
            code = lsb.FIELD[field]
            assert g.lib.lsb_get_fields(g.h, 0, code, level, ctypes.c_void_p(small.data_ptr()), nb - 1, 0) == 1
    g.close()
