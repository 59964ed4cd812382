"""The one-launch depth stage of short lists: bit-exact order at its edges (one key, whole and partial
thread rows, the longest short list and the first long one), with tied and culled particles."""
import numpy as np
import pytest
import torch  # noqa: F401

import oracle
from gpu_helpers import run_gpu, to_np
from paper_2412_12507_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("n", [1, 31, 33, 1023, 1024, 1025, 7169, 8191, 8192, 8193])
@pytest.mark.parametrize("depths", ["spread", "tied", "equal"])
@pytest.mark.parametrize("W,H,tw,th", [(70, 33, 16, 16), (1100, 1000, 8, 8)])  # 15 and 17250 tiles
def test_short_lists_bit_exact(n, depths, W, H, tw, th):
    rect, depth = synth.random_rects(n, n, W, H, max_w=30, max_h=20)
    if depths == "tied":
        depth = np.round(depth, 1).astype(np.float32)
    elif depths == "equal":  # every digit alike: no pass runs, the index order is the result
        depth = np.full_like(depth, 2.5)
        rect = np.maximum(rect, 0)
    cam = synth.camera("pinhole", W, H, fx=float(W))
    g = run_gpu(synth.scene_cube(n, 1), cam, synth.options(tile_w=tw, tile_h=th), want_keys=True, rect=rect, depth=depth)
    k_ref, v_ref, r_ref = oracle.bin_keys(depth, rect, W, H, tw, th)
    K, b = g["K"], g["binning"]
    assert K == len(k_ref) == g["K_sum"]
    assert np.array_equal(to_np(b.keys)[:K].view(np.uint64), k_ref)
    assert np.array_equal(to_np(b.vals)[:K].view(np.uint32), v_ref)
    assert np.array_equal(to_np(b.ranges).view(np.uint32), r_ref)
