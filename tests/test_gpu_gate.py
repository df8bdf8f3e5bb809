"""The records of several cameras against those of one camera after another (other
kernels), and the gate's bulk copies against its plain loads, around the sizes of
its chunks: 128 Gaussians or candidates, 16 or 64 chunks per block."""
import dataclasses

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


def _scene(n, lod):
    g = synth.plain_scene(n, seed=n)
    rng = np.random.default_rng(n + 1)
    if lod:
        g = dataclasses.replace(g, lod=rng.integers(0, 6, n).astype(np.uint8))
    return B.GaussianTensors.from_host(g)


def _cameras(k):
    cams = []
    for q in range(k):
        c = synth.plain_camera(64 + 16 * (q % 5), 48 + 16 * (q % 3), 60.0 + 8 * q)
        t = np.array([0.2 * np.sin(q), 0.1 * q / k, 0.3 * np.cos(q)], np.float32)
        cams.append(dataclasses.replace(c, t=t, campos=-t)) # R is the identity
    return cams


def _records(g, cams, params, slots):
    ws = B.Workspace(max_gaussians=g.n, max_records=slots, max_instances=64 * slots, max_tiles=4096,
                     max_pixels=1 << 20, max_cameras=len(cams))
    ws.preprocess(g, cams, params)
    ws.bin_sort()
    ws.sync_status()
    c = ws.counts()
    n = c["n_records"]
    r = lambda which, dtype, k: ws.read_buffer(which, dtype, n, k).reshape(n, k)
    ints = np.concatenate([r(B.GS_BUF_REC_GAUSSIAN, np.uint32, 1), r(B.GS_BUF_REC_RECT, np.uint32, 2),
                           r(B.GS_BUF_REC_TILES, np.uint32, 1), r(B.GS_BUF_REC_DEPTH, np.uint32, 1)], 1)
    floats = np.concatenate([r(B.GS_BUF_REC_XY_CONIC, np.float32, 4), r(B.GS_BUF_REC_C_OPAC_RG, np.float32, 4),
                             r(B.GS_BUF_REC_B_LO, np.float32, 4)], 1)
    return r(B.GS_BUF_REC_CAMERA, np.uint16, 1)[:, 0], ints, floats, c


PARAMS = {False: B.RenderParams(), True: B.RenderParams(lod_enable=True, lod_d0=2.5, lod_f=1.25, lod_Lmax=5)}


@pytest.mark.parametrize("lod", [False, True])
@pytest.mark.parametrize("n,k", [(1, 2), (2, 64), (127, 3), (128, 2), (129, 24), (2047, 5), (2049, 64), (8193, 3),
                                 (90_000, 2)])
def test_several_cameras_as_one_after_another(n, k, lod):
    g, cams = _scene(n, lod), _cameras(k)
    cam, ints, floats, c = _records(g, cams, PARAMS[lod], n * k)
    total = tiles = 0
    visible = np.zeros(n, bool)
    for q in range(k):
        _, i1, f1, c1 = _records(g, [cams[q]], PARAMS[lod], n)
        assert np.array_equal(ints[cam == q], i1), q
        # the same arithmetic, contracted by the compiler as it likes: a few units
        # in the last place of values up to the image's size
        assert np.allclose(floats[cam == q], f1, rtol=1e-4, atol=1e-4), q
        total += len(i1)
        tiles += c1["instances_needed"]
        visible[i1[:, 0]] = True
    assert len(cam) == total and c["instances_needed"] == tiles and c["n_visible"] == visible.sum()
    order = ints[:, 0].astype(np.int64) * 64 + cam
    assert np.all(np.diff(order) > 0) # (Gaussian, camera) order


@pytest.mark.parametrize("k", [1, 3])
@pytest.mark.parametrize("n", [1, 15, 127, 128, 129, 1025, 8192, 82_000])
def test_unaligned_labels_take_the_plain_loads(n, k):
    g, cams = _scene(n, True), _cameras(k)
    lod = torch.empty(n + 1, dtype=torch.uint8, device="cuda")
    lod[1:] = g.lod
    shifted = dataclasses.replace(g, lod=lod[1:])
    assert shifted.lod.data_ptr() % 16
    a, b = _records(g, cams, PARAMS[True], n * k), _records(shifted, cams, PARAMS[True], n * k)
    for x, y in zip(a[:3], b[:3]):
        assert np.array_equal(x, y)
    assert a[3] == b[3]
