"""The record buffers of a pass (trace_kappa, trace_shear, trace_method_a,
trace_tiles), without a GPU: a tracer that launches nothing, over buffers that
hold no memory (torch's meta device)."""
import contextlib
import weakref

import numpy as np
import pytest

import synth


class Buffers:
    """torch.empty and torch.cuda.stream, watched: the live buffers' records,
    their peak, and the stream that each was allocated for."""

    def __init__(self, monkeypatch):
        import torch
        self.live = self.peak = 0
        self.streams, self.current = [], None
        empty = torch.empty

        def watched(*size, **kw):
            t = empty(*size, **kw)
            if t.device.type == "meta" and t.dim() == 2:
                self.streams.append(self.current)
                self.live += t.shape[0]
                self.peak = max(self.peak, self.live)
                weakref.finalize(t, self._drop, t.shape[0])
            return t

        @contextlib.contextmanager
        def on(stream):
            before, self.current = self.current, stream
            yield
            self.current = before

        monkeypatch.setattr(torch, "empty", watched)
        monkeypatch.setattr(torch.cuda, "stream", on)
        monkeypatch.setattr(torch.cuda, "Stream", Stream)

    def _drop(self, n):
        self.live -= n


class Stream:
    cuda_stream = 1234


@pytest.fixture
def rrp(monkeypatch):
    import paper_1601_02012_gb300 as pkg
    from paper_1601_02012_gb300 import build
    build.build()

    class Tracer(pkg.Tracer):
        def __init__(self, bundle, method_a=False, shear=False, fp64_dda=False):
            self.method_a, self.generic = method_a, False
            self.desc = pkg._rr.bundle_desc(bundle, method_a=method_a, shear=shear, fp64_dda=fp64_dda)
            self.boxes = []

        def set_observer(self, obs):
            self.desc.obs[:] = obs

        def tidal(self, *args, **kw):
            pass

        def tidal_box(self, grid, phi, rec, bbox, delta=None, stream=None):
            self.boxes.append(bbox)
            assert rec.shape[0] == pkg._points(bbox) < 2 ** 31

        def steps(self, grid, recs, steps, boxes=None, stream=None):
            assert len(recs) == len(steps) and (boxes is None or len(boxes) == len(steps))

        step = tidal

        def finalize(self, stream=None):
            return None, None

        def shear(self, stream=None):
            return None, None

        def segments(self):
            return 0

        def close(self):
            pass

    monkeypatch.setattr(pkg, "Tracer", Tracer)
    return pkg


def _steps(b, n):
    cuts = np.linspace(b.chi_s, 0.0, n + 1)
    return [synth.Step(float(x), float(y), 1.0, 1.0) for x, y in zip(cuts[:-1], cuts[1:])]


@pytest.mark.parametrize("call", ["kappa", "whole", "shear", "method_a", "tiles"])
def test_records_belong_to_the_stream(rrp, monkeypatch, call):
    """A pass drops its buffers while the stream still reads them: every one is
    allocated for the stream that the pass runs on, so that no other stream's
    work is given the memory."""
    import torch
    g = synth.Grid((64, 64, 64), 64.0)
    b = synth.Bundle(8, 8, synth.deg(5), synth.deg(5), (32.0, 32.0, 0.0), 60.0)
    phi = torch.empty(g.n, device="meta")
    watch, s = Buffers(monkeypatch), Stream()
    steps = _steps(b, 20)
    if call == "tiles":
        rrp.trace_tiles([(phi, g, b.obs)] * 3, b, steps, stream=s)
    elif call in ("kappa", "whole"):
        rrp.trace_kappa(phi, g, b, steps, footprint=call == "kappa", stream=s)
    else:
        getattr(rrp, "trace_" + call)(phi, g, b, steps, stream=s)
    assert watch.streams and all(x is s for x in watch.streams)


@pytest.mark.parametrize("call", ["kappa", "shear"])
def test_boxes_past_32_bits(rrp, call):
    """Steps whose own boxes hold 2^31 points or more, which box-local records
    do not take, run on whole-grid records."""
    import torch
    g = synth.Grid((2048, 2048, 2048), 2048.0)
    b = synth.Bundle(8, 8, synth.deg(50), synth.deg(50), (1024.0, 1024.0, 2.0), 2000.0)
    getattr(rrp, "trace_" + call)(torch.empty(g.n, device="meta"), g, b, _steps(b, 2))


@pytest.mark.parametrize("call", ["kappa", "shear", "method_a", "tiles"])
@pytest.mark.parametrize("n,depth,steps,fov", [(512, 10.0, 40, 5.0), (512, 18.0, 72, 3.0), (64, 1.0, 16, 40.0),
                                               (512, 0.97, 40, 10.0)])
def test_no_more_than_a_whole_grid(rrp, monkeypatch, call, n, depth, steps, fov):
    """A pass never holds more records than a whole grid has, also where the
    cone passes through many periods and each step has a box of its own."""
    import torch
    g = synth.Grid((n, n, n), float(n))
    b = synth.Bundle(64, 64, synth.deg(fov), synth.deg(fov), (0.5 * n, 0.5 * n, 1.0), depth * n)
    phi = torch.empty(g.n, device="meta")
    watch = Buffers(monkeypatch)
    if call == "tiles":
        rrp.trace_tiles([(phi, g, b.obs)] * 2, b, _steps(b, steps))
    else:
        getattr(rrp, "trace_" + call)(phi, g, b, _steps(b, steps))
    assert 0 < watch.peak <= g.ncells and watch.live == 0
