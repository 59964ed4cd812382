"""bin_and_sort at the edges of its rules on sizes: the two-launch passes' group of 16 radix tiles
(32,768 particles), their limit of 1024 radix tiles for the depth sort (2,097,152 particles) and for the
column sort (2,097,152 keys of capacity), every combination of both, and group totals that do not fit
the row stage's spine (few tile rows).  Bit-exact against a stable sort by (tile, depth bits, index)."""
import numpy as np
import pytest
import torch

from gpu_helpers import to_np
from paper_2412_12507_gb300 import render, synth

pytestmark = pytest.mark.gpu

LIMIT = 1 << 21


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _lists(rect, depth, live, tiles_x, tw, th):
    """(keys, vals) of the live particles' tiles, sorted stably by (tile, depth bits, index)."""
    idx = np.flatnonzero(live)
    r = rect[idx].astype(np.int64)
    c0, c1, r0, r1 = r[:, 0] // tw, r[:, 2] // tw, r[:, 1] // th, r[:, 3] // th
    keys, vals = [], []
    for dy in range(int((r1 - r0).max()) + 1):
        for dx in range(int((c1 - c0).max()) + 1):
            m = (r0 + dy <= r1) & (c0 + dx <= c1)
            tile = ((r0 + dy) * tiles_x + c0 + dx)[m].astype(np.uint64)
            keys.append((tile << np.uint64(32)) | depth[idx[m]].view(np.uint32).astype(np.uint64))
            vals.append(idx[m])
    keys, vals = np.concatenate(keys), np.concatenate(vals)
    o = np.lexsort((vals, keys))
    return keys[o], vals[o].astype(np.uint32)


def _check(n, capacity, W, H, n_live, tw=16, th=16):
    rng = np.random.default_rng(n + capacity)
    x0, y0 = rng.integers(0, W, n), rng.integers(0, H, n)
    rect = np.stack([x0, y0, np.minimum(x0 + rng.integers(0, 24, n), W - 1),
                     np.minimum(y0 + rng.integers(0, 24, n), H - 1)], axis=1).astype(np.int16)
    live = np.zeros(n, bool)
    live[rng.choice(n, n_live, replace=False)] = True
    depth = (1.0 + np.round(rng.random(n) * 1000) / 100).astype(np.float32)  # many ties
    rect[~live] = (0, 0, -1, -1)
    r = rect.astype(np.int64)
    nt = np.where(live, (r[:, 2] // tw - r[:, 0] // tw + 1) * (r[:, 3] // th - r[:, 1] // th + 1), 0)
    cam, op = synth.camera("pinhole", W, H, fx=float(W)), synth.options(tile_w=tw, tile_h=th)
    d = lambda a: torch.as_tensor(a).cuda()  # noqa: E731
    proj = render.Projection(None, None, d(depth), d(rect), d(nt.astype(np.int32)))
    K = int(nt.sum())
    assert K <= capacity
    b = render.bin_and_sort(proj, cam, op, capacity, want_keys=True)
    keys, vals = _lists(rect, depth, live, -(-W // tw), tw, th)
    assert b.count() == K == len(keys)
    assert np.array_equal(to_np(b.keys[:K]).view(np.uint64), keys)
    assert np.array_equal(to_np(b.vals[:K]).view(np.uint32), vals)
    tile = (keys >> np.uint64(32)).astype(np.int64)
    T = render.tile_count(cam, op)
    start, end = np.searchsorted(tile, np.arange(T)), np.searchsorted(tile, np.arange(T), side="right")
    ranges = to_np(b.ranges).view(np.uint32)
    full = start < end
    assert np.array_equal(ranges[full], np.stack([start, end], 1)[full])
    assert (ranges[~full, 0] == ranges[~full, 1]).all()


@pytest.mark.parametrize("capacity", [LIMIT, LIMIT + 1])
@pytest.mark.parametrize("n", [8193, 32768, 32769, LIMIT, LIMIT + 1])
def test_pass_limits(n, capacity):
    _check(n, capacity, 1000, 700, min(n, 200_000))


@pytest.mark.parametrize("capacity", [32768, 32769, LIMIT, LIMIT + 1])
@pytest.mark.parametrize("n", [8192, 32769, 1_300_000])
def test_few_tile_rows(n, capacity):
    """One row of 40 tiles: 1.3 million particles' group totals outgrow the row stage's spine."""
    _check(n, capacity, 640, 16, 8000)


@pytest.mark.parametrize("n", [8192, 32769, LIMIT + 1])
def test_more_than_256_columns(n):
    _check(n, LIMIT, 4200, 64, min(n, 100_000))
