"""The row copies of compaction and density control at the edges of their
paths: sizes around the block and chunk sizes, arrays that are not 16-byte
aligned, models without moments, and outputs that do not fit."""
import numpy as np
import pytest
import torch

from paper_2605_13794_gb300 import binding as B
from paper_2605_13794_gb300 import synth

pytestmark = pytest.mark.gpu

NAMES = ("mean", "log_scale", "quat", "opacity_logit", "sh")
SHAPES = dict(mean=(3,), log_scale=(3,), quat=(4,), opacity_logit=(), sh=(16, 3))


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2605_13794_gb300 import build
    build.build()


def _rows(n, gen, pad):
    """Rows of every parameter in storage that starts `pad` floats into an allocation."""
    def one(shape):
        k = int(np.prod(shape, dtype=int))
        return torch.randn(n * k + pad, generator=gen, device="cuda")[pad:].view(n, *shape)
    return B.GaussianTensors(*[one(SHAPES[k]) for k in NAMES], None)


def _model(n, pad=0, moments=True, seed=3):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    g = _rows(n, gen, pad)
    g.lod = torch.randint(0, 6, (n,), generator=gen, device="cuda", dtype=torch.uint8)
    return B.ModelTensors(g, _rows(n, gen, pad) if moments else None, _rows(n, gen, pad) if moments else None)


def _ws(n):
    return B.Workspace(max_gaussians=n, max_records=1, max_instances=1, max_tiles=1, max_pixels=1, model_ops=True)


@pytest.mark.parametrize("n", [1, 3, 255, 256, 257, 2049])
@pytest.mark.parametrize("src_pad,dst_pad", [(0, 0), (1, 0), (0, 1), (3, 2)])
def test_compaction_of_unaligned_rows(n, src_pad, dst_pad):
    src, dst = _model(n, src_pad), _model(n, dst_pad, seed=4)
    keep = np.random.default_rng(n).uniform(size=n) < 0.6
    n_out = torch.zeros(1, dtype=torch.int64, device="cuda")
    ws = _ws(n)
    ws.compact(src, torch.from_numpy(synth.pack_bits(keep).view(np.int32)).cuda(), dst, n_out)
    ws.sync_status()
    k = int(keep.sum())
    assert int(n_out) == k
    at = torch.from_numpy(keep).cuda()
    untouched = _model(n, dst_pad, seed=4)
    for part in ("g", "m", "v"):
        for name in NAMES:
            got = getattr(getattr(dst, part), name)
            assert torch.equal(got[:k], getattr(getattr(src, part), name)[at]), (part, name)
            assert torch.equal(got[k:], getattr(getattr(untouched, part), name)[k:]), (part, name)
    assert torch.equal(dst.g.lod[:k], src.g.lod[at])


@pytest.mark.parametrize("pad", [0, 1])
@pytest.mark.parametrize("short", [0, 1, 2, 5])
def test_density_control_into_too_few_rows(pad, short):
    """Every Gaussian cloned: 2n rows.  A shorter output keeps the pairs that fit whole, leaves
    the rest alone and reports the capacity."""
    n = 301
    src = _model(n, pad)
    src.g.opacity_logit.fill_(1.0)
    src.g.log_scale.fill_(-9.0)
    rows = 2 * n - short
    dst, before = _model(rows, pad, seed=5), _model(rows, pad, seed=5)
    one = torch.ones(n, dtype=torch.int32, device="cuda")
    n_out = torch.zeros(1, dtype=torch.int64, device="cuda")
    ws = _ws(n)
    ws.densify(src, torch.ones(n, device="cuda"), one, one, one, torch.zeros(n, 2, 3, device="cuda"), dst, n_out)
    if short:
        with pytest.raises(B.GSError) as e:
            ws.sync_status()
        assert e.value.code == B.GS_ERR_CAPACITY
    else:
        ws.sync_status()
    assert int(n_out) == 2 * n
    fit = rows // 2
    for name in NAMES:
        got, ref = getattr(dst.g, name), getattr(src.g, name)
        assert torch.equal(got[0:2 * fit:2], ref[:fit]) and torch.equal(got[1:2 * fit:2], ref[:fit]), name
        assert torch.equal(got[2 * fit:], getattr(before.g, name)[2 * fit:]), name
        for part in ("m", "v"):
            mom = getattr(getattr(dst, part), name)
            assert torch.equal(mom[0:2 * fit:2], getattr(getattr(src, part), name)[:fit]), (part, name)
            assert not mom[1:2 * fit:2].any(), (part, name)
    assert torch.equal(dst.g.lod[0:2 * fit:2], src.g.lod[:fit])


def test_moments_that_are_not_carried_start_from_zero():
    n = 1000
    src, dst = _model(n, moments=False), _model(n)
    keep = torch.full(((n + 31) // 32,), -1, dtype=torch.int32, device="cuda")
    n_out = torch.zeros(1, dtype=torch.int64, device="cuda")
    ws = _ws(n)
    ws.compact(src, keep, dst, n_out)
    ws.sync_status()
    for name in NAMES:
        assert torch.equal(getattr(dst.g, name), getattr(src.g, name))
        assert not getattr(dst.m, name).any() and not getattr(dst.v, name).any()
