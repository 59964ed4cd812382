"""Renderer.forward's host copy of the key count does not depend on the torch modes that are on when a
renderer is first used: a renderer warmed up in inference mode trains afterwards, and one made under a
default device renders."""
import pytest
import torch

from paper_2412_12507_gb300 import render, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _default_device():
    return torch.device("cuda")


@pytest.mark.parametrize("mode", [torch.inference_mode, torch.no_grad, _default_device])
def test_first_use_under_a_mode(mode):
    case = synth.small_pinhole(seed=0, n=300)
    cam, op = case["camera"], case["options"]
    scene = render.Scene.from_arrays(case["scene"])
    ref = render.Renderer(cam, op).forward(scene).rgb.clone()
    r = render.Renderer(cam, op)
    with mode():
        assert torch.equal(r.forward(scene).rgb, ref)
    assert torch.equal(r.forward(scene).rgb, ref)
    with mode():
        assert torch.equal(r.forward(scene).rgb, ref)
    leaves = [t.clone().requires_grad_(True) for t in (scene.means, scene.log_scales, scene.quats,
                                                       scene.opacity_logits, scene.sh)]
    rgb, alpha = render.render(*leaves, scene.sh_degree, r)
    (rgb.sum() + alpha.sum()).backward()
    assert torch.equal(rgb.detach(), ref) and all(torch.isfinite(t.grad).all() for t in leaves)
