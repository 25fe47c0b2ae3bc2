"""GPU tests of what a batched step costs beside its tiles: the launch's CTAs past the tile table, and
how the tiles of a small batch are spread over the chip. Times are the least of several runs; each
bound lies between two measured behaviours."""
import time

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


def _batch(lbm, sizes, running=None, **kw):
    b = lbm.Batch(sizes, **W.MODEL, **kw)
    mu = W.MODEL["k2"] * lbm.lbm_coexistence(W.MODEL["eos"], W.MODEL["Tr"])["mu_sat"]
    for i, (nx, ny) in enumerate(sizes[:running]):
        R = float(max(6, min(nx, ny) // 4))
        b.set_geometry(i, circle=(nx // 2 + 0.0, 0.0, R), mu_circle=mu, mu_bottom=mu, mu_top=mu,
                       drop=(nx // 2 + 0.0, R + 0.3 * ny, 0.15 * ny, 5.6))
    return b


def _us_per_step(b, steps=400, runs=8):
    best = float("inf")
    for _ in range(runs):
        t = time.perf_counter()
        b.run(steps, check_every=steps, tol=0.0)
        best = min(best, time.perf_counter() - t)
    return best / steps * 1e6


def test_ctas_past_the_tile_table_leave_at_once(lbm):
    """One running lattice in a batch of 64 (20,480 CTAs per step, 320 with a tile): 13 us per step when
    the others leave after reading the table's length, 21 us when each first releases the next launch."""
    b = _batch(lbm, [(512, 320)] * 64, running=1)
    us = _us_per_step(b)
    b.close()
    assert us < 18.0, us


def test_tiles_of_a_small_batch_are_spread_over_the_chip(lbm):
    """528 tiles of 32x16 against 704: three to four tiles per SM against five. Evenly spread the first
    take 0.89 of the second's time, crowded 0.98."""
    us = []
    for sizes in ([(230, 340)] * 3, [(110, 345)] * 8):
        b = _batch(lbm, sizes)
        us.append(_us_per_step(b, steps=1000))
        b.close()
    assert us[0] < 0.95 * us[1], us


@pytest.mark.parametrize("auto", [False, True])
def test_autotuning_keeps_the_form_of_small_batches(lbm, auto):
    """Two 96x64 lattices run in 320-thread tiles of 16x8, which the tuner has to time as well: tuned
    (by hand or at the first run) the batch is no slower than untuned, where the 256-thread variants
    take 1.5 times as long. The entries keep their order and number."""
    sizes = [(96, 64)] * 2
    plain, tuned = _batch(lbm, sizes), _batch(lbm, sizes, tile_auto=auto)
    if not auto:
        res = tuned.autotune(20)
        tiles = [(32, 8), (32, 16), (64, 16), (32, 32)]
        assert [(r["tile"], r["persistent"]) for r in res] == [(t, p) for t in tiles for p in (False, True)]
        assert min(res, key=lambda r: r["us_per_step"])["tile"] == (32, 16)
    a, b = _us_per_step(plain, steps=1000), _us_per_step(tuned, steps=1000)
    plain.close()
    tuned.close()
    assert b < 1.15 * a, (a, b)
