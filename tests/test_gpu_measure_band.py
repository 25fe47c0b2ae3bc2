"""GPU tests of the one-kernel reductions and of the measurement's two node sets: rows that end
inside an eight-node access, the list of nodes near the wall against the whole-lattice scan, and
the batched residual's sums against exactly rounded host sums."""
import math

import numpy as np
import pytest

from helpers import gpu_lattice, oracle_config
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


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nx,ny", [(8, 9), (9, 8), (15, 40), (257, 33), (2056, 11), (30, 1300)])
def test_mass_of_ragged_rows(lbm, nx, ny, precision):
    """Flat walls, random densities: mass within 4 ulp-sized steps of the exactly rounded sum (a
    tree of FP64 additions over at most 2^6 partial sums per thread keeps log-depth error; 1e-15
    relative is above it), liquid count and centroid exactly."""
    rng = np.random.default_rng(nx * 1000 + ny)
    rho = rng.uniform(0.05, 8.1, size=(ny, nx)).astype(np.float32).astype(np.float64)
    lat = lbm.Lattice(nx, ny, **W.MODEL, precision=precision)
    lat.set_geometry(rho0=rho)
    info = lat.info()
    got = lat.mass()
    liq = rho > 0.5 * (info.rho_g + info.rho_l)
    jj, ii = np.nonzero(liq)
    assert got["mass"] == pytest.approx(math.fsum(rho.ravel().tolist()), rel=1e-15, abs=0)
    assert got["n_liquid"] == liq.sum()
    assert got["cx"] == float(ii.sum()) / len(ii) and got["cy"] == float(jj.sum()) / len(jj)
    lat.close()


@pytest.mark.parametrize("R", [60.0, 900000.0, 1100000.0])
def test_listed_and_scanned_nodes_give_the_oracle_angles(lbm, oracle_mod, R):
    """A drop on a cylinder whose top is at y = 20: R = 1.1e6 lies outside the range of the node
    list, so the measurement scans the lattice; links, points and distances equal the oracle's
    on the identical field in every case."""
    O = oracle_mod
    w = W.Workload("band", 180, 110, (90.0, 20.0 - R, R),
                   (90.0, 20.5 + 12.0, 30.0, 10.0))
    cfg = oracle_config(O, w)[0]
    rho = O.Sim(cfg).rho().astype(np.float32).astype(np.float64)
    lat = gpu_lattice(lbm, cfg, rho0=rho)
    l, r = lat.measure()
    ol, orr, _ = O.measure(cfg, rho, 0.5 * (cfg.rho_g + cfg.rho_l))
    for g, o in ((l, ol), (r, orr)):
        assert g.status == 0 and o.status == 0
        assert (g.link1, g.link2) == (o.link1, o.link2)
        assert g.d1 == o.d1 and g.d2 == o.d2
        assert abs(g.theta - o.theta) < 1e-6
    lat.close()


def test_batch_residual_matches_host_sums(lbm):
    """Residual of a batched run against sums of the same two fields on the host (all terms of
    one sign: 1e-13 is far above the rounding of either side)."""
    sizes = [(96, 64), (77, 53), (203, 41)]
    b = lbm.Batch(sizes, **W.MODEL)
    for i, (nx, ny) in enumerate(sizes):
        b.set_geometry(i, circle=(nx // 2, 0.0, 15.0), drop=(nx // 2 + 0.0, 25.0, 10.0, 5.6))
    b.run(20, check_every=20, tol=0.0)
    before = [b.rho(i) for i in range(len(sizes))]
    _, _, res = b.run(20, check_every=20, tol=0.0)
    for i in range(len(sizes)):
        after = b.rho(i)
        want = math.fsum(np.abs(after - before[i]).ravel().tolist()) / math.fsum(after.ravel().tolist())
        assert res[i] == pytest.approx(want, rel=1e-13, abs=0)
    b.close()


@pytest.mark.parametrize("R,lift,r,side", [(20.0, 0.0, 12.0, -1), (20.0, 0.0, 17.3, 1),
                                           (24.5, 0.5, 10.0, -1), (35.0, 0.0, 14.0, 1),
                                           (35.0, 0.5, 12.0, -1), (28.0, 0.3, 13.0, 1)])
def test_links_between_nearly_equal_densities(lbm, oracle_mod, R, lift, r, side):
    """FP64 lattices almost uniform at rho_m: the two densities are one FP32 spacing apart and rho_m lies
    0.49 spacings from an FP32 number, so that a point placed with FP32 densities sits at the end of its
    link (up to 0.9 of a link away). The chosen links, distances and angles equal the oracle's on the
    identical field; in most of these cases the FP32 point of a chosen link lies outside the band."""
    O = oracle_mod
    nx, ny = 120, 90
    w = W.Workload("flat", nx, ny, (60.0, 0.0, R), (60.0, R + 0.6 * r + lift, r, 5.6))
    cfg = oracle_config(O, w)[0]
    mid = np.float32(0.5 * (cfg.rho_g + cfg.rho_l))
    ulp = float(np.spacing(mid))
    cfg.rho_l = 2 * (float(mid) + side * 0.49 * ulp) - cfg.rho_g
    rho_m = 0.5 * (cfg.rho_g + cfg.rho_l)
    jj, ii = np.mgrid[0:ny, 0:nx]
    low, high = (0.9, 0.1) if side > 0 else (0.1, 0.9)
    rho = np.where(np.hypot(ii - w.drop[0], jj - w.drop[1]) < r, rho_m + high * ulp, rho_m - low * ulp)
    lat = gpu_lattice(lbm, cfg, precision=1, rho0=rho)
    ol, orr, _ = O.measure(cfg, rho, rho_m)
    for g, o in zip(lat.measure(), (ol, orr)):
        assert g.status == 0 and o.status == 0
        assert (g.link1, g.link2) == (o.link1, o.link2)
        assert g.d1 == o.d1 and g.d2 == o.d2
        assert abs(g.theta - o.theta) < 1e-6
    lat.close()
