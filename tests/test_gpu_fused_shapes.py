"""Gradients after the fused walk on every tile shape: the entries that it notes for
the adjoint are those that the forward alone notes, with and without marked records."""
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


@pytest.mark.parametrize("cull", [False, True])
@pytest.mark.parametrize("tw,th", [(16, 16), (32, 8), (8, 32), (32, 16), (16, 8), (8, 16)])
def test_the_adjoint_after_the_fused_walk(tw, th, cull):
    n, cam = 12_000, synth.plain_camera(203, 149, 190.0)
    host = synth.plain_scene(n, seed=71)
    host.opacity_logit[: n // 2] += 4.0  # pixels that stop early and pixels that do not
    g = B.GaussianTensors.from_host(host)
    params = B.RenderParams(tile_w=tw, tile_h=th, cull_enable=B.GS_CULL_MARK if cull else B.GS_CULL_OFF)
    words = torch.from_numpy(synth.random_cull_bits(n, 0.4, 5).view(np.int32)).cuda() if cull else None
    P = cam.width * cam.height
    dL = torch.randn(3 * P, generator=torch.Generator(device="cuda").manual_seed(7), device="cuda")
    out = []
    for fused in (False, True):
        ws = B.Workspace(max_gaussians=n, max_records=n, max_instances=64 * n, max_tiles=B.tiles_of(cam, tw, th),
                         max_pixels=P)
        ws.preprocess(g, [cam], params, words)
        ws.bin_sort()
        rgb, T = torch.empty(3 * P, device="cuda"), torch.empty(P, device="cuda")
        (ws.render_fwd_importance if fused else ws.render_fwd)(rgb, T)
        grads = g.zeros_like()
        ws.render_bwd(g, dL, grads)
        ws.sync_status()
        out.append([rgb, T] + grads.params())
        ws.close()
    for a, b in zip(*out):
        assert torch.equal(a, b)
    assert all(bool(t.abs().max() > 0) for t in out[0][2:])
