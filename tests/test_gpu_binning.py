"""Tile lists of every length class of the per-tile sort, against a sort of the
library's own records by (depth bits, record): exact."""
import numpy as np
import pytest
import torch

from paper_2605_13794_gb300 import binding as B
from paper_2605_13794_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2605_13794_gb300 import build
    build.build()


def _scene(n, seed, spread):
    """Small Gaussians in front of the camera; every third depth occurs twice or more."""
    g = synth.plain_scene(n, seed=seed)
    rng = np.random.default_rng(seed)
    g.mean[:, :2] *= spread
    g.mean[::3, 2] = 2.0 + rng.integers(0, max(n // 8, 1), len(g.mean[::3])) / 64.0
    return B.GaussianTensors.from_host(g)


def _check(ws, cam, instances):
    c = ws.counts()
    n = c["n_records"]
    depth = ws.read_buffer(B.GS_BUF_REC_DEPTH, np.uint32, n)
    rect = ws.read_buffer(B.GS_BUF_REC_RECT, np.uint32, n, 2)
    tx = (cam.width + 15) // 16
    tiles = tx * ((cam.height + 15) // 16)
    ranges = ws.read_buffer(B.GS_BUF_TILE_RANGES, np.uint32, tiles, 2)
    vals = ws.read_buffer(B.GS_BUF_SORTED_VALUES, np.uint32, min(c["n_instances"], instances))
    x0, y0, x1, y1 = rect[:, 0] & 0xFFFF, rect[:, 0] >> 16, rect[:, 1] & 0xFFFF, rect[:, 1] >> 16
    order = np.lexsort((np.arange(n), depth))
    longest = 0
    for t in range(tiles):
        x, y = t % tx, t // tx
        ref = order[(x0[order] <= x) & (x < x1[order]) & (y0[order] <= y) & (y < y1[order])]
        s, e = ranges[t]
        assert np.array_equal(vals[s:e], ref), t
        longest = max(longest, len(ref))
    return longest


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 64, 65, 128, 129, 255, 257, 512, 513, 1024, 1025, 2047, 2048, 2049,
                               4096, 4097, 6145, 9000])
def test_one_tile_of_every_length(n):
    cam = synth.plain_camera(16, 16, 20.0)
    g = _scene(n, 100 + n, 0.02)
    ws = B.Workspace(max_gaussians=n, max_records=n, max_instances=n, max_tiles=1, max_pixels=256)
    for _ in range(2):  # the second pass finds the counts and look-back words cleared
        ws.preprocess(g, [cam], B.RenderParams())
        ws.bin_sort()
        ws.bin_sort()   # the same binning again
        ws.sync_status()
        assert _check(ws, cam, n) == n


def test_lists_of_mixed_lengths():
    n = 30_000
    cam = synth.plain_camera(150, 90, 120.0)
    g = _scene(n, 7, 0.35)
    ws = B.Workspace(max_gaussians=n, max_records=n, max_instances=16 * n, max_tiles=64, max_pixels=150 * 90)
    ws.preprocess(g, [cam], B.RenderParams())
    ws.bin_sort()
    ws.sync_status()
    assert _check(ws, cam, 16 * n) > 2048


def test_too_few_instances_is_reported_and_the_next_binning_is_whole():
    n = 3000
    cam = synth.plain_camera(64, 48, 80.0)
    g, few = _scene(n, 8, 0.2), _scene(200, 9, 0.2)
    ws = B.Workspace(max_gaussians=n, max_records=n, max_instances=2500, max_tiles=12, max_pixels=64 * 48)
    ws.preprocess(g, [cam], B.RenderParams())
    ws.bin_sort()
    with pytest.raises(B.GSError) as e:
        ws.sync_status()
    assert e.value.code == B.GS_ERR_CAPACITY
    assert ws.counts()["n_instances"] == 2500 and ws.counts()["instances_needed"] > 2500
    ws.clear_error()
    ws.preprocess(few, [cam], B.RenderParams())
    ws.bin_sort()
    ws.sync_status()
    _check(ws, cam, 2500)
    torch.cuda.synchronize()


@pytest.mark.parametrize("depths", ["near", "wide", "pairs", "equal"])
@pytest.mark.parametrize("n", [2, 31, 33, 64, 127, 128, 129, 255, 256, 257, 511, 1025, 2048, 4100])
def test_depths_that_fit_a_sort_word_and_those_that_do_not(n, depths):
    """Distinct depths in one binade (their bits fit beside the place), over eight
    decades (cut bits: distinct or clashing), a single equal pair, all equal."""
    cam = synth.plain_camera(16, 16, 20.0)
    g = synth.plain_scene(n, seed=n)
    rng = np.random.default_rng(n)
    z = 4.0 + rng.permutation(n).astype(np.float32) * np.float32(3.0 / n)
    if depths == "wide":
        z = 10.0 ** rng.uniform(0.0, 8.0, n)
    elif depths == "pairs":
        z[-1] = z[0]
    elif depths == "equal":
        z[:] = 5.0
    g.mean[:, :2] = 0.0
    g.mean[:, 2] = z
    ws = B.Workspace(max_gaussians=n, max_records=n, max_instances=n, max_tiles=1, max_pixels=256)
    ws.preprocess(B.GaussianTensors.from_host(g), [cam], B.RenderParams())
    ws.bin_sort()
    ws.sync_status()
    assert _check(ws, cam, n) == n
