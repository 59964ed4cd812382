"""The k-buffer backward's SH gradients over the whole range of their weights: infinite ones stay the
infinities (and the sums of both signs the NaN) that FP32 products give, and the relative accuracy does
not depend on the loss's scale."""
import numpy as np
import pytest
import torch

from gpu_helpers import to_np
from paper_2412_12507_gb300 import render, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _sh_grads(deg, up):
    """dL/dsh of two particles that every pixel of a 16 x 16 image blends, colours positive."""
    rng = np.random.default_rng(1)
    scene = render.Scene.from_arrays(dict(
        means=np.array([[0, 0, 3], [0.1, 0, 3.5]], np.float32), log_scales=np.zeros((2, 3), np.float32),
        quats=np.tile(np.array([1, 0, 0, 0], np.float32), (2, 1)), opacity_logits=np.zeros(2, np.float32),
        sh=np.abs(0.02 * rng.standard_normal((2, (deg + 1) ** 2, 3))).astype(np.float32), sh_degree=deg))
    cam, op = synth.camera("pinhole", 16, 16, fx=32.0, fy=32.0), synth.options(kbuffer=4)
    r = render.Renderer(cam, op, capacity=1 << 12)
    f = r.forward(scene)
    assert (f.alpha > 0.1).all()
    g = r.backward(scene, up, torch.zeros_like(f.alpha))
    return to_np(g["sh"]).astype(np.float64)


@pytest.mark.parametrize("deg", [0, 1, 2, 3])
def test_infinite_weights(deg):
    up = torch.zeros((3, 16, 16), device="cuda")
    up[0, 3, 5] = float("inf")   # one pixel of one channel
    up[1] = float("inf")         # all of another
    g = _sh_grads(deg, up)
    assert np.isposinf(g[:, 0, :2]).all() and (g[:, :, 2] == 0).all()
    assert not np.isfinite(g[:, :, :2]).any()
    up[1, :, ::2] = float("-inf")
    g = _sh_grads(deg, up)
    assert np.isposinf(g[:, 0, 0]).all() and np.isnan(g[:, :, 1]).all()


@pytest.mark.parametrize("deg", [0, 1, 2, 3])
@pytest.mark.parametrize("y,x", [(3, 5), (15, 0)])
def test_accuracy_over_the_losss_scale(deg, y, x):
    """One pixel's gradient, so that no sum hides a product's rounding.  Scaling the loss by a power of
    two scales every weight exactly; a product of two 24-bit operands, through six cross terms or
    directly, is within 4 x 2^-24 of the exact one on either side, and results that a global
    reduction flushes (subnormal ones) are below 2^-126 / 2^-99 of the largest."""
    ref = None
    for e in (0, -50, -62, -80, -96, 100):
        up = torch.zeros((3, 16, 16), device="cuda")
        up[:, y, x] = torch.tensor([0.7, -1.3, 0.9], device="cuda") * 2.0 ** e
        g = _sh_grads(deg, up) * 2.0 ** -e
        ref = g if ref is None else ref
        assert np.abs(g - ref).max() <= 8 * 2.0 ** -24 * np.abs(ref).max(), e
