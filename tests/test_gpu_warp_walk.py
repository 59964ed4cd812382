"""The tile-order compositing kernels walk a tile with independent warps of 64 pixels: the edges of
that walk's chunks of list entries, of its pixel layouts and of its aligned copies."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import TOL, compare_frame, grad_compare, run_gpu, to_np
from paper_2412_12507_gb300 import render, synth

pytestmark = pytest.mark.gpu

# one warp (8x8), squares with a ragged image, two 8x4 blocks with an empty second half (8x12),
# row-major with an unfilled last warp (12x8), five warps in two blocks (20x16), eight in two (16x32)
TILES = [(8, 8), (16, 16), (8, 12), (12, 8), (20, 16), (16, 32), (64, 1)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _list_case(n, deg, rs):
    """n broad, faint particles in front of a small ragged image: every tile lists all of them, and
    no pixel saturates."""
    sc = synth.scene_cube(n, 40 + n, log_s=(-0.7, 0.2), logit_std=0.1, deg=deg, lo=(-.5, -.5, 2.5), hi=(.5, .5, 3.5))
    sc["opacity_logits"] = sc["opacity_logits"] - np.float32(3.5)
    kw = {}
    if rs:
        qe, te = synth.rs_end_pose(0.05, 2.0)
        kw = dict(q_end=qe, t_end=te, rolling_shutter=1)
    return sc, synth.camera("fisheye" if rs else "pinhole", 37, 29, fx=30.0, fy=30.0, **kw)


@pytest.mark.parametrize("n", [1, 24, 25, 32, 33, 64, 65])
@pytest.mark.parametrize("deg,rs", [(0, 0), (2, 1), (3, 0)])
def test_chunk_edges_render_matches_oracle(n, deg, rs):
    sc, cam = _list_case(n, deg, rs)
    op = synth.options()
    ref = oracle.render(sc, cam, op, tol=TOL)
    g = run_gpu(sc, cam, op)
    r = compare_frame(g["frame"], ref)
    assert r["n_bad"] == 0, r
    assert g["K"] >= 4 * n  # four of the six tiles list every particle


@pytest.mark.parametrize("mode", [{}, dict(colour_mode=1), dict(kernel_degree=3)])
def test_pixel_layouts_give_identical_images(mode):
    """Every layout of the pixels over warps, and rows of SH coefficients without 16-byte alignment,
    give the bits of the 16 x 16 tiles."""
    sc = synth.scene_cube(700, 5, log_s=(-3.0, 0.6), deg=3)
    cam = synth.camera("fisheye", 101, 67, k=(0.02, -0.01, 0.0, 0.0))
    ref = None
    for tw, th in TILES:
        f = run_gpu(sc, cam, synth.options(tile_w=tw, tile_h=th, **mode))["frame"]
        img = [to_np(t) for t in (f.rgb, f.alpha, f.t_final)]
        if ref is None:
            ref = img
        assert all(np.array_equal(a, b) for a, b in zip(img, ref)), (tw, th)
    op = synth.options(**mode)
    g = run_gpu(sc, cam, op)
    s = g["scene"]
    sh = torch.empty(s.sh.numel() + 1, device="cuda")[1:].view_as(s.sh).copy_(s.sh)
    assert sh.data_ptr() % 16 == 4
    f = render.composite_forward(render.Scene(s.means, s.log_scales, s.quats, s.opacity_logits, sh, 3), cam, op,
                                 g["proj"], g["binning"])
    assert np.array_equal(to_np(f.rgb), ref[0])


def _oracle_grads(sc, cam, op, seed):
    W, H = cam["width"], cam["height"]
    proj = oracle.project(sc, cam, op, TOL)
    f = oracle.render(sc, cam, op, proj=proj, tol=TOL)
    ok = (f["flags"] & oracle.F_BACKWARD_TIES) == 0  # zero upstream where the decisions may differ
    rng = np.random.default_rng(seed)
    w_rgb, w_a = rng.standard_normal((H * W, 3)) * ok[:, None], rng.standard_normal(H * W) * ok
    ref = oracle.backward(sc, cam, op, proj, (f["px"], f["py"]), w_rgb, w_a, magnitudes=True)
    up = [torch.as_tensor(a.astype(np.float32)).cuda() for a in (w_rgb.T.reshape(3, H, W), w_a.reshape(H, W))]
    return ref, up


def _check_grads(g, cam, op, up, ref):
    grads = render.composite_backward(g["scene"], cam, op, g["proj"], g["binning"], g["frame"], *up)
    for k in ("means", "log_scales", "quats", "opacity_logits", "sh"):
        grad_compare(to_np(grads[k]), ref[k], ref["mag"][k], k)
    return grads


@pytest.mark.parametrize("n", [1, 24, 25, 32, 33, 65])
@pytest.mark.parametrize("deg,rs,mode", [(3, 1, {}), (2, 0, {}), (3, 0, dict(colour_mode=1)), (1, 1, dict(colour_mode=1))])
def test_chunk_edges_backward_matches_oracle(n, deg, rs, mode):
    sc, cam = _list_case(n, deg, rs)
    op = synth.options(**mode)
    ref, up = _oracle_grads(sc, cam, op, n)
    _check_grads(run_gpu(sc, cam, op), cam, op, up, ref)


@pytest.mark.parametrize("mode", [{}, dict(colour_mode=1)])
def test_pixel_layouts_backward_matches_oracle(mode):
    """Every layout of the pixels over warps; and gradient rows without 16-byte alignment, written
    to by the C entry, agree with the aligned ones to the reductions' rounding."""
    sc = synth.scene_cube(300, 6, log_s=(-2.8, 0.5), deg=3)
    cam = synth.camera("pinhole", 61, 45, fx=55.0, fy=55.0)
    ref, up = _oracle_grads(sc, cam, synth.options(**mode), 9)
    for tw, th in TILES:
        op = synth.options(tile_w=tw, tile_h=th, **mode)
        g = run_gpu(sc, cam, op)
        _check_grads(g, cam, op, up, ref)
    empty_like = torch.empty_like
    try:
        render.torch.empty_like = lambda t: torch.empty(t.numel() + 1, device="cuda")[1:].view_as(t) if t.dim() == 3 \
            else empty_like(t)
        grads = _check_grads(g, cam, op, up, ref)
        assert grads["sh"].data_ptr() % 16 == 4
    finally:
        render.torch.empty_like = empty_like


def test_infinite_upstream_stays_with_its_pixel():
    """A pixel with an infinite upstream gradient, or a particle with infinite SH coefficients, reaches
    only the particles that pixel blends, and pixels that particle covers: a thread's other pixel keeps
    its own finite sums."""
    mk = lambda x, y: [x, y, 3.0]  # noqa: E731
    sc = synth.scene_cube(2, 3, deg=1)
    sc["means"] = np.array([mk(-0.10, -0.406), mk(-0.10, -0.156)], np.float32)  # rows 4 apart in one warp
    sc["log_scales"] = np.full((2, 3), -3.6, np.float32)
    sc["opacity_logits"] = np.zeros(2, np.float32)
    cam = synth.camera("pinhole", 16, 16, fx=48.0, fy=48.0)
    op = synth.options()
    g = run_gpu(sc, cam, op)
    r = to_np(g["proj"].rect)
    assert r[0][3] < r[1][1]  # disjoint rows
    up = [torch.ones((3, 16, 16), device="cuda"), torch.zeros((16, 16), device="cuda")]
    fin = render.composite_backward(g["scene"], cam, op, g["proj"], g["binning"], g["frame"], *up)
    up[0][:, : r[0][3] + 1] = float("inf")
    out = render.composite_backward(g["scene"], cam, op, g["proj"], g["binning"], g["frame"], *up)
    for k in fin:
        assert not torch.isfinite(out[k][0]).all() and torch.equal(out[k][1], fin[k][1]), k
    s = g["scene"]
    s.sh[0, 0] = float("inf")
    f = render.composite_forward(s, cam, op, g["proj"], g["binning"])
    keep = torch.ones((16, 16), dtype=torch.bool, device="cuda")
    keep[r[0][1]:r[0][3] + 1, r[0][0]:r[0][2] + 1] = False
    assert torch.equal(f.rgb[:, keep], g["frame"].rgb[:, keep]) and not torch.isfinite(f.rgb).all()
