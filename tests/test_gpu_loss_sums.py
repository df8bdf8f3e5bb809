"""The partial sums of the loss: exact where the pixels' sum over a warp is."""
import numpy as np
import pytest
import torch

from paper_2605_13794_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2605_13794_gb300 import build
    build.build()


# The L1 term alone (lambda 0) of images that differ by v everywhere.  v has 21
# significant bits, so up to eight of it add exactly in FP32, and a warp's 32 such
# sums do: the mean is v to the last bit.  1152 v, a tile of 36 rows, needs 25 bits.
@pytest.mark.parametrize("views,h,w", [(1, 64, 64), (2, 576, 640), (1, 1152, 1088)])
def test_a_constant_difference_is_its_own_mean(views, h, w):
    v = np.float32((round(0.95 * 2**21) | 1) / 2**21)
    x = torch.full((views, 3, h, w), float(v), device="cuda")
    y = torch.zeros_like(x)
    ws = B.Workspace(max_gaussians=1, max_records=1, max_instances=1, max_tiles=1, max_pixels=views * h * w)
    loss, dL = torch.zeros(1, device="cuda"), torch.empty_like(x)
    ws.photometric_loss(x, y, 0.0, loss, dL)
    torch.cuda.synchronize()
    assert loss.item() == float(v)
