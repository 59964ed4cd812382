"""Renderer.forward reads the key count back while the compositing is already queued: a call whose keys
do not fit renders again, and returns the frame, the binning and the gradients of the second pass."""
import pytest
import torch

from paper_2412_12507_gb300 import render, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("kbuffer", [0, 4])
def test_overflow_renders_again(kbuffer):
    case = synth.rs_fisheye(n=3000, width=203, height=117)
    cam, op = case["camera"], dict(case["options"], kbuffer=kbuffer)
    scene = render.Scene.from_arrays(case["scene"])
    wide = render.Renderer(cam, op)
    a = wide.forward(scene)
    K = wide.binning.count()
    for capacity in (1, K - 1, K):
        r = render.Renderer(cam, op, capacity=capacity)
        for _ in range(2):  # the second frame fits at once
            b = r.forward(scene)
            assert r.binning.count() == K <= r.binning.capacity
            assert all(torch.equal(getattr(a, f), getattr(b, f)) for f in ("rgb", "alpha", "t_final", "n_used"))
        assert r.capacity == (capacity if capacity == K else int(K * r.growth) + 1)
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            b = r.forward(scene)
        side.synchronize()
        assert torch.equal(a.rgb, b.rgb)
