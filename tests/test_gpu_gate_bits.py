"""The records of several cameras against those of one camera after another: what
explicitly rounded operations give is the same bit for bit, the low words of the
means included; opacity and colour agree to their rounding."""
import numpy as np
import pytest

from paper_2605_13794_gb300 import binding as B
from paper_2605_13794_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2605_13794_gb300 import build
    build.build()


def _cameras(k):
    cams = []
    for q in range(k):
        eye = (0.3 * np.sin(q), 0.1 * np.cos(2 * q), -0.2 * q / k)
        cams.append(synth.look_at_camera(eye, (0.0, 0.1 * np.sin(q), 4.0), (0.0, -1.0, 0.0), 1000 + 16 * q, 700, 40.0 + q))
    return cams


def _records(g, cams, slots):
    ws = B.Workspace(max_gaussians=g.n, max_records=slots, max_instances=256 * slots,
                     max_tiles=sum(B.tiles_of(c) for c in cams), max_pixels=sum(c.width * c.height for c in cams),
                     max_cameras=len(cams))
    ws.preprocess(g, cams, B.RenderParams())
    ws.bin_sort()
    ws.sync_status()
    n = ws.counts()["n_records"]
    rd = np.concatenate([ws.read_buffer(w, np.float32, n, 4) for w in
                         (B.GS_BUF_REC_XY_CONIC, B.GS_BUF_REC_C_OPAC_RG, B.GS_BUF_REC_B_LO)], 1)
    cam = ws.read_buffer(B.GS_BUF_REC_CAMERA, np.uint16, n)
    who = ws.read_buffer(B.GS_BUF_REC_GAUSSIAN, np.uint32, n)
    ws.close()
    return cam, who, rd


@pytest.mark.parametrize("n,k", [(129, 24), (5000, 2), (5000, 5)])
def test_the_same_records_bit_for_bit(n, k):
    g = B.GaussianTensors.from_host(synth.plain_scene(n, seed=n))
    cams = _cameras(k)
    cam, who, rd = _records(g, cams, n * k)
    low = 0
    for q in range(k):
        _, who1, rd1 = _records(g, [cams[q]], n)
        got = rd[cam == q]
        assert np.array_equal(who[cam == q], who1)
        # u, v, A, k; D; u_lo, v_lo and the mark
        for at in (0, 1, 2, 3, 4, 9, 10, 11):
            assert np.array_equal(got[:, at].view(np.uint32), rd1[:, at].view(np.uint32)), (q, at)
        low += np.count_nonzero(rd1[:, 9]) + np.count_nonzero(rd1[:, 10])
        # opacity; colour: 16 terms of at most about 1 each, 2^-23 of a sum of at most 16
        for at in (5, 6, 7, 8):
            assert np.abs(got[:, at] - rd1[:, at]).max() <= 2e-6, (q, at)
    assert low > len(who)  # most low words are not zero
