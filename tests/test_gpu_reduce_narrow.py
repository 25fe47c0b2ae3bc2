"""GPU tests of the reduction on lattices of more rows than the reduction has blocks, whose blocks take
several rows at once where a row needs few threads."""
import time

import numpy as np
import pytest

from helpers import tanh_drop
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


def _lattice(lbm, nx, ny, rho, precision=0):
    co = lbm.lbm_coexistence(W.MODEL["eos"], W.MODEL["Tr"])
    mu = W.MODEL["k2"] * co["mu_sat"]
    lat = lbm.Lattice(nx, ny, **W.MODEL, precision=precision)
    lat.set_geometry(mu_bottom=mu, mu_top=mu, rho0=rho, drop=(nx / 2, ny / 2, 5.0, 5.6))
    return lat


# rows beside the 1216 blocks of a chip with 152 SMs, columns around 8 x a power of two threads
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nx,ny", [(8, 1216), (8, 1217), (9, 2433), (16, 9731), (17, 4865), (33, 1300),
                                   (130, 2500), (1025, 1300), (8, 311297)])
def test_sums_of_tall_lattices(lbm, nx, ny, precision):
    if precision and ny > 100000:
        pytest.skip("the FP32 case covers the stride")
    co = lbm.lbm_coexistence(W.MODEL["eos"], W.MODEL["Tr"])
    rho = tanh_drop(nx, ny, nx / 2, 0.6 * ny, 40.0, co["rho_g"], co["rho_l"], 5.6)
    rho *= 1 + 1e-3 * np.sin(0.1 * np.arange(ny))[:, None]
    rho = rho.astype(np.float32).astype(np.float64)
    lat = _lattice(lbm, nx, ny, rho, precision)
    m = lat.mass()
    liquid = rho > 0.5 * (co["rho_g"] + co["rho_l"])
    j, i = np.nonzero(liquid)
    # FP64 sums of at most 2.5 M positive values in any order: relative error below 1e-12 with room
    assert abs(m["mass"] - rho.sum()) <= 1e-12 * rho.sum()
    assert int(m["n_liquid"]) == liquid.sum()
    assert abs(m["cx"] - i.mean()) <= 1e-9 * nx and abs(m["cy"] - j.mean()) <= 1e-9 * ny
    lat.close()


def test_narrow_lattices_take_no_longer(lbm):
    """The sums of 8 x 100000 against those of 100 x 8000: the same number of nodes. With one row per block
    2.4 times the time, with as many rows as threads fit close to 1; the bound lies between."""
    us = []
    for nx, ny in ((100, 8000), (8, 100000)):
        lat = _lattice(lbm, nx, ny, np.full((ny, nx), 0.5))
        best = float("inf")
        for _ in range(30):
            t = time.perf_counter()
            lat.mass()
            best = min(best, time.perf_counter() - t)
        us.append(best * 1e6)
        lat.close()
    assert us[1] < 1.7 * us[0], us
