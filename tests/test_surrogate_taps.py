"""Every tap of every convolution's gradients, on the lattices of test_gpu_surrogate_wide.py. There the
initial weights make pre-activations of both signs, FP32 arithmetic alone moves gradients by percents
and the bounds have to be as wide. Here each output channel copies two of the 9 C_in inputs (plus a
small positive rest), inputs are noise in (0.2, 1) and biases positive: pre-activations stay positive,
activations keep their differences from pixel to pixel through all levels, and FP32 arithmetic moves
the gradients by 2e-4 at most, while two taps in each other's place move them by 1e-3 and more."""
import numpy as np
import pytest

import test_gpu_surrogate as T
from test_gpu_surrogate import env  # noqa: F401  (fixture)

SHAPES = [(8, 16, 128, 2), (16, 16, 128, 2), (16, 24, 256, 2), (16, 40, 384, 1), (32, 24, 128, 2),
          (32, 16, 256, 1), (32, 16, 192, 2)]  # base, H, W, images


def _case(base, H, Wd, B):
    from oracle import surrogate as S
    rng = np.random.default_rng(base * 1000 + Wd)
    x = rng.uniform(0.2, 1.0, size=(B, H, Wd, 8)).astype(np.float32)
    t = rng.uniform(0, 1, size=(B, H, Wd)).astype(np.float32)
    m = (rng.uniform(size=(B, H, Wd)) > 0.3).astype(np.uint8)
    convs, n = S.layer_specs(base)
    p, o = np.zeros(n, np.float32), 0
    for ci, co, _ in convs:
        w = rng.uniform(0, 0.3 / (9 * ci), size=(co, 9, ci))
        for _ in range(2):
            w[np.arange(co), rng.integers(0, 9, co), rng.integers(0, ci, co)] += 0.5
        p[o:o + w.size] = w.ravel()
        o += w.size
        p[o:o + co] = 0.02
        o += co
    p[o:o + base] = rng.normal(0, 1.0, base)
    return x, t, m, p


def _reference(x, t, m, p, base):
    """The oracle's gradients with BF16 storage, and per layer the bound: eight times what the same
    network evaluated in FP32 departs from FP64, at least 4e-4."""
    import torch
    from oracle import surrogate as S
    pw, xb = T._bf16(p), T._bf16(x)
    layers, head = T._layers(base)
    for sw, sb in layers:
        pw[sb] = p[sb]
    pw[head] = p[head]
    rec = []
    S.forward(torch.tensor(pw), torch.tensor(xb), base, bf16_activations=True, record=rec)
    assert min(float(z.min()) for z in rec) > 0.01  # far from the kink against BF16 rounding
    _, g, _ = S.loss_and_grad(pw, xb, t.astype(np.float64), m.astype(bool), base, True, True)
    g32 = T._fp32_yardstick(pw, xb, t, m, base)
    bounds = [max(4e-4, 8 * max(T._rel(g32[k], g[k]) for k in pair)) for pair in layers]
    return g, layers, head, bounds


@pytest.mark.parametrize("base,H,Wd,B", SHAPES)
def test_swapped_taps_exceed_the_bounds(base, H, Wd, B):
    """On the CPU: of every layer's weight gradient, any two taps exchanged (left and right, a tap and
    its neighbour, above and below) leave the bound of the GPU test behind."""
    from oracle import surrogate as S
    x, t, m, p = _case(base, H, Wd, B)
    g, layers, _, bounds = _reference(x, t, m, p, base)
    for k, ((ci, co, _), (sw, _)) in enumerate(zip(S.layer_specs(base)[0], layers)):
        w = g[sw].reshape(co, 9, ci)
        for a, b in ((3, 5), (4, 5), (3, 4), (0, 1), (0, 2), (1, 7), (6, 8)):
            v = w.copy()
            v[:, [a, b]] = v[:, [b, a]]
            assert np.linalg.norm(v - w) / np.linalg.norm(w) > 1.5 * bounds[k], (k, a, b)


@pytest.mark.gpu
@pytest.mark.parametrize("base,H,Wd,B", SHAPES)
def test_gradients_tap_by_tap(env, base, H, Wd, B):  # noqa: F811
    x, t, m, p = _case(base, H, Wd, B)
    g, layers, head, bounds = _reference(x, t, m, p, base)
    gpu, _, _, _ = T._gpu_and_oracle(env, x, t, m, p, base, H, Wd)
    for k, pair in enumerate(layers):
        for s in pair:
            assert T._rel(gpu["g"][s], g[s]) < bounds[k], (k, T._rel(gpu["g"][s], g[s]), bounds[k])
    assert T._rel(gpu["g"][head], g[head]) < 1e-3
