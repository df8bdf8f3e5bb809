"""The loss at image sizes around the edges of its tiles (32 columns; 32 rows, or 36
in the forward of many tiles), against the float64 oracle."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2605_13794_gb300 import binding as B
from tests.gpu_helpers import assert_grad_close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2605_13794_gb300 import build
    build.build()
    O.build()


# tolerances: FP32 sums of 121 products of values up to 1 and a quotient, as for
# any other size
@pytest.mark.parametrize("views,h,w", [(1, 1, 1), (1, 1, 40), (1, 40, 1), (1, 5, 6), (2, 31, 31), (1, 32, 33), (1, 35, 32),
                                       (1, 36, 32), (3, 37, 33), (1, 41, 27), (1, 64, 64), (1, 71, 65), (1, 72, 31),
                                       (2, 73, 96), (1, 108, 97),
                                       # more tiles than are resident at once: the forward's 36 rows
                                       (4, 71, 900), (4, 72, 897), (4, 73, 899), (7, 37, 900), (2, 109, 1500)])
def test_sizes_around_the_tile_edges(views, h, w):
    rng = np.random.default_rng(1000 * h + w)
    x = rng.uniform(0, 1, (views, 3, h, w)).astype(np.float32)
    y = rng.uniform(0, 1, (views, 3, h, w)).astype(np.float32)
    ws = B.Workspace(max_gaussians=1, max_records=1, max_instances=1, max_tiles=64, max_cameras=1, max_pixels=views * h * w)
    xt, yt = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    loss, dL = torch.zeros(1, device="cuda"), torch.empty_like(xt)
    ws.photometric_loss(xt, yt, 0.2, loss, dL)
    torch.cuda.synchronize()
    ref, grad = O.photometric_loss(x, y, lam=float(np.float32(0.2)))
    assert abs(loss.item() - ref) <= 1e-5 * abs(ref)
    assert_grad_close("dL/dimage", dL.double().cpu().numpy(), grad, rtol=1e-3)
