"""A captured one-camera pass replayed with more cameras in the table takes the first."""
import dataclasses

import pytest
import torch

from paper_2605_13794_gb300 import binding as B
from paper_2605_13794_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2605_13794_gb300 import build
    build.build()


@pytest.mark.parametrize("more", [1, 63])
@pytest.mark.parametrize("n", [100, 3000])
def test_one_camera_graph_with_a_longer_table(n, more):
    g, params = B.GaussianTensors.from_host(synth.plain_scene(n, seed=17)), B.RenderParams()
    first = synth.plain_camera(96, 80, 110.0)
    other = dataclasses.replace(first, fx=140.0, fy=140.0)
    ws = B.Workspace(max_gaussians=n, max_records=n, max_instances=64 * n, max_tiles=64 * 30, max_pixels=64 * 96 * 80,
                     max_cameras=64)
    rgb, T = torch.empty(3 * 96 * 80, device="cuda"), torch.empty(96 * 80, device="cuda")

    def rest():
        ws.preprocess_uploaded(g, params)
        ws.bin_sort()
        ws.render_fwd(rgb, T)

    ws.upload_cameras([other], params)
    rest()
    ws.sync_status()
    want = rgb.clone(), T.clone()
    ws.upload_cameras([first], params)
    rest()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        rest()
    ws.upload_cameras([other] + [first] * more, params)
    graph.replay()
    ws.sync_status()
    assert torch.equal(rgb, want[0]) and torch.equal(T, want[1])
