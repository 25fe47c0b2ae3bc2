"""Lattices whose rows are wide enough for the surrogate kernels that stage operand rows: the first
convolution and its weight gradient (rows of 128 pixels), the marching convolutions (128) and the
weight gradients from staged rows (64), at the smallest heights, at ragged widths and with images of
which a tile is the whole, against the oracle that stores activations and gradients in BF16."""
import numpy as np
import pytest

import test_gpu_surrogate as T
from test_gpu_surrogate import env  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("base,H,Wd,B", [(8, 16, 128, 2), (16, 8, 128, 1), (16, 16, 128, 2),
                                         (16, 40, 384, 1), (16, 24, 256, 2), (32, 24, 128, 2), (32, 16, 256, 1),
                                         (32, 16, 192, 2)])
def test_wide_rows_match_oracle(env, base, H, Wd, B):  # noqa: F811
    """Seeded initial weights. Forward and loss within BF16 storage of the oracle. Pre-activations
    within a rounding step of the leaky ReLU's kink flip with any FP32-level difference, so the
    gradients are compared by direction, layer by layer; the bound is four times what the same
    network evaluated in FP32 on the CPU departs from its FP64 evaluation (at least 1e-2 per layer and
    1e-3 for the whole gradient). Reading a layer's taps in the wrong order gives cosines of 0.24-0.97."""
    x, t, m, p = T._case(base=base, H=H, Wd=Wd, B=B)
    gpu, ref, pw, xb = T._gpu_and_oracle(env, x, t, m, p, base, H, Wd)
    full = ref["full"]
    assert np.abs(gpu["phi"] - full["phi"]).max() < 1e-3
    assert gpu["loss"] == pytest.approx(full["loss"], rel=1e-4)
    g32 = T._fp32_yardstick(pw, xb, t, m, base)
    layers, head = T._layers(base)
    worst = max(1 - T._cos(g32[k], full["g"][k]) for pair in layers for k in pair)
    for k, pair in enumerate(layers):
        for sl in pair:
            assert 1 - T._cos(gpu["g"][sl], full["g"][sl]) < max(1e-2, 4 * worst), k
    assert 1 - T._cos(gpu["g"], full["g"]) < max(1e-3, 4 * (1 - T._cos(g32, full["g"])))
    assert T._rel(gpu["g"][head], full["g"][head]) < 2e-2
