"""autograd.Renderer called from several streams: one context serves one render at a
time, so a render on another stream has to wait for the last one, on the device. The
order is checked on the host with recorded calls, the images on the GPU."""
import types

import numpy as np
import pytest
import torch

from paper_2501_01628_gb300 import autograd, synth


@pytest.mark.parametrize("handles", [(5, 7), (0, 7), (5, 0)])  # 0: the default stream
def test_a_render_on_another_stream_waits_for_the_last_one(monkeypatch, handles):
    log, state = [], dict(stream=None, capturing=False)

    class Stream:
        def __init__(self, name, handle):
            self.name, self.cuda_stream = name, handle

        def wait_event(self, event):
            log.append("%s waits for %s" % (self.name, event.at))

        def wait_stream(self, other):
            assert other.cuda_stream == 0  # any other may be gone
            log.append("%s waits for %s" % (self.name, other.name))

    class Event:
        def record(self, stream):
            self.at = stream.name

    calls = {name: (lambda name: lambda *a, **k: log.append("%s %s" % (state["stream"].name, name)))(name)
             for name in ("vr_create", "vr_set_render_params", "vr_render_frame", "vr_render_backward", "vr_sync",
                          "vr_destroy")}
    a, b = Stream("a", handles[0]), Stream("b", handles[1])
    state["stream"] = a
    monkeypatch.setattr(autograd, "vr", types.SimpleNamespace(**calls))
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *_: state["stream"])
    monkeypatch.setattr(torch.cuda, "Event", Event)
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: state["capturing"])
    monkeypatch.setattr(autograd.Renderer, "_bind", lambda self, tf, density, cam, stream=None: log.append(
        "%s bind" % state["stream"].name))
    r = autograd.Renderer(dict(kind="grid", grid=(1, 1, 1)), 0.0, 1.0, device=0)
    tf, density = torch.zeros((2, 4), requires_grad=True), torch.zeros((2, 2, 2), requires_grad=True)

    def render(stream):
        state["stream"] = stream
        del log[:]
        img = r.render(tf, density, dict(height=2, width=3))
        return img, list(log)

    assert render(a)[1] == ["a bind", "a vr_render_frame"]
    assert render(a)[1] == ["a bind", "a vr_render_frame"]
    img, calls_b = render(b)
    assert calls_b == ["b waits for a", "b bind", "b vr_render_frame"]
    state["stream"] = a
    del log[:]
    autograd._Render.backward(img.grad_fn, torch.zeros((2, 3, 4)))
    assert log == ["a waits for b", "a bind", "a vr_render_backward", "a vr_sync"]
    assert render(b)[1] == ["b bind", "b vr_render_frame"]  # the backward is known to be done
    state["capturing"] = True  # events of a capture and of outside don't mix
    assert render(a)[1] == ["a bind", "a vr_render_frame"]


@pytest.mark.gpu
def test_images_from_alternating_streams():
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    rng = np.random.default_rng(4)
    vol = torch.from_numpy(synth.blob_volume(128, synth.draw_blobs(rng, 8))).cuda()
    tables = [torch.from_numpy(synth.random_tf(rng, alpha_max=0.05)).cuda() for _ in range(3)]
    cams = [synth.orbit_camera(400, 300, az) for az in (10.0, 130.0, 250.0)]
    r = autograd.Renderer(dict(kind="grid", grid=(2, 2, 2)), 0.0, 1.5)
    try:
        want = []
        for tf, cam in zip(tables, cams):
            want.append(r.render(tf, vol, cam))
            torch.cuda.synchronize()
        streams = [torch.cuda.current_stream(), torch.cuda.Stream(), torch.cuda.Stream()]
        got = []
        torch.cuda.synchronize()
        for k in range(30):
            with torch.cuda.stream(streams[(k * 7 // 3) % 3]):
                got.append((k % 3, r.render(tables[k % 3], vol, cams[k % 3])))
        torch.cuda.synchronize()
        for k, img in got:
            assert torch.equal(img, want[k])
    finally:
        r.close()
