"""GPU tests of the field read-out on lattices of every width: values, and that a narrow lattice is read as
quickly as a wide one of as many nodes."""
import time

import numpy as np
import pytest

from paper_2202_06516_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_2202_06516_gb300 import lbm as L
    L.lib()
    return L


# widths around the powers of two that a block's rows are split by, and past one column block
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nx,ny", [(8, 8), (9, 301), (17, 64), (64, 33), (130, 21), (1023, 9), (1025, 10),
                                   (2051, 8)])
def test_read_back_equals_the_start(lbm, nx, ny, precision):
    """The density read back is the FP32-representable one that was set, at fluid nodes; 0 in the solid."""
    rng = np.random.default_rng(nx)
    rho = rng.uniform(0.05, 8.1, size=(ny, nx)).astype(np.float32).astype(np.float64)
    lat = lbm.Lattice(nx, ny, **W.MODEL, precision=precision)
    R = 3.0
    lat.set_geometry(circle=(nx // 2 + 0.0, 0.0, R), rho0=rho)
    jj, ii = np.mgrid[0:ny, 0:nx]
    solid = (ii - nx // 2) ** 2 + jj ** 2 <= R * R
    assert np.array_equal(lat.rho(), np.where(solid, 0.0, rho))
    lat.close()


def test_narrow_lattices_read_as_quickly_as_wide_ones(lbm):
    """16 x 60000 against 1024 x 938, as many nodes: with a row per block the narrow one took 2.4 times as long."""
    import torch
    us = []
    for nx, ny in ((16, 60000), (1024, 938)):
        lat = lbm.Lattice(nx, ny, **W.MODEL)
        lat.set_geometry(drop=(nx / 2, 20.0, 5.0, 5.6))
        out = torch.empty(ny, nx, dtype=torch.float64, device="cuda")
        best = float("inf")
        for _ in range(30):
            t = time.perf_counter()
            lbm.lbm_read_fields(lat.ctx, lbm.LBM_FIELD_RHO, nx, ny, device_out=(out.data_ptr(), None, None))
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t)
        us.append(best * 1e6)
        lat.close()
    assert us[0] < 1.5 * us[1], us
