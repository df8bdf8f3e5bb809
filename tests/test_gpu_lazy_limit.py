"""Deferred Adam steps at the end of their history: a step past max_steps is
refused and reported, and changes nothing."""
import numpy as np
import pytest
import torch

from paper_2605_13794_gb300 import binding as B
from paper_2605_13794_gb300 import synth
from paper_2605_13794_gb300.train import TrainStep

pytestmark = pytest.mark.gpu

LR = [1.6e-3, 5e-3, 1e-3, 5e-2, 2.5e-3]
W, H = 96, 80


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2605_13794_gb300 import build
    build.build()


def _view(k):
    cam = synth.look_at_camera((0.5 * k, 0.1, 0.2 * k), (0.3 * k - 0.3, 0.0, 4.0), (0.0, -1.0, 0.0), W, H, 35.0)
    target = torch.from_numpy(synth.noise_target(W, H, seed=40 + k)[None].astype(np.float32)).cuda()
    return [cam], target


def _training(max_steps):
    ts = TrainStep(B.GaussianTensors.from_host(synth.plain_scene(4000, seed=91)), *_view(0), B.RenderParams(), LR,
                   lazy=True)
    ts.ws.adam_lazy_enable(ts.m, ts.v, ts.last, ts.drift, max_steps=max_steps)
    for k in range(2):
        ts.set_views(*_view(k))
        ts.run()
    ts.ws.sync_status()
    return ts


def _state(ts):
    ts.flush()
    torch.cuda.synchronize()
    return ts.g.params() + ts.m.params() + ts.v.params() + [ts.last, ts.drift]


@pytest.mark.parametrize("graph", [False, True])
def test_a_step_past_the_history_is_refused(graph):
    ref, ts = _training(1000), _training(2)
    if graph:
        ts.capture()
    for k in (2, 0): # a new view, whose candidates are brought up to date, and one seen before
        ts.set_views(*_view(k))
        ts.replay() if graph else ts.run()
        with pytest.raises(B.GSError) as e:
            ts.ws.sync_status()
        assert e.value.code == B.GS_ERR_CAPACITY
    with pytest.raises(B.GSError) as e: # the step's number given: refused by the call
        ts.run(step=3)
    assert e.value.code == B.GS_ERR_CAPACITY
    for a, b in zip(_state(ref), _state(ts)):
        assert torch.equal(a, b)
    assert int(ts.last.min()) == int(ts.last.max()) == 2
    # with a longer history the training goes on where it stopped
    ts.ws.adam_lazy_enable(ts.m, ts.v, ts.last, ts.drift, max_steps=1000)
    for t in (ref, ts):
        t.set_views(*_view(2))
        t.run()
        t.ws.sync_status()
    for a, b in zip(_state(ref), _state(ts)):
        assert torch.equal(a, b)
    assert int(ts.last.max()) == 3


def test_no_step_is_taken_when_the_steps_are_deferred_after_the_preprocess():
    # every Gaussian with a record is behind when the step is refused
    ts = _training(2)
    before = [t.clone() for t in _state(ts)]
    ws = ts.ws
    ws.adam_lazy_disable()
    ws.preprocess_uploaded(ts.g, ts.params)
    ws.bin_sort()
    ws.render_fwd(ts.rgb)
    ts.dL.normal_()
    ws.render_bwd_compact(ts.g, ts.dL)
    ts.last.zero_()
    ws.adam_lazy_enable(ts.m, ts.v, ts.last, ts.drift, max_steps=1)
    ws.adam_step_compact(ts.g, ts.m, ts.v, LR, 0)
    with pytest.raises(B.GSError) as e:
        ws.sync_status()
    assert e.value.code == B.GS_ERR_CAPACITY
    before[-2].zero_()
    for a, b in zip(before, ts.g.params() + ts.m.params() + ts.v.params() + [ts.last, ts.drift]):
        assert torch.equal(a, b)
