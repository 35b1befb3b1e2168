"""A pass on a stream that is not torch's current one: its record buffers are
dropped with its steps still queued, and other work is not given their memory."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rrp():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1601_02012_gb300 import build
    build.build()
    import paper_1601_02012_gb300 as pkg
    return pkg


@pytest.mark.parametrize("raw", [False, True])
def test_tiles_beside_other_work(rrp, monkeypatch, raw):
    """While a tile's trace waits on a side stream, with its records computed,
    the default stream allocates buffers of their size and fills them with NaN:
    the maps stay those of a pass with nothing beside it."""
    import torch
    g = synth.Grid((36, 44, 70), 46.8)
    depth = g.n[2] * g.h
    b = synth.Bundle(37, 22, synth.deg(11), synth.deg(8), (23.4, 28.6, 0.0), 2.9 * depth, periodic=False)
    cuts = np.linspace(b.chi_s, 0.0, 13)
    steps = [synth.Step(float(x), float(y), 1.0, 0.9) for x, y in zip(cuts[:-1], cuts[1:])]
    phi = torch.from_numpy(synth.random_field(g.n, 6, np.float32)).cuda()
    obs = [(b.obs[0], b.obs[1], -i * depth) for i in range(3)]
    want = rrp.trace_tiles([(phi, g, o) for o in obs], b, steps)
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    recorded = []
    trace = rrp.Tracer.steps

    def slow(self, *args, **kw):
        recorded.append(torch.cuda.Event())
        recorded[-1].record(s)
        with torch.cuda.stream(s):
            torch.cuda._sleep(200_000_000)   # about 0.1 s
        trace(self, *args, **kw)

    monkeypatch.setattr(rrp.Tracer, "steps", slow)

    def tiles():
        for o in obs:
            if recorded:
                recorded[-1].synchronize()
                other = [torch.full((g.ncells, 8), float("nan"), device="cuda") for _ in range(3)]
                torch.cuda.default_stream().synchronize()
                del other
            yield phi, g, o

    got = rrp.trace_tiles(tiles(), b, steps, stream=s.cuda_stream if raw else s)
    assert len(recorded) == 3 and got[2] == want[2]
    for x, y in zip(got[:2], want[:2]):
        assert torch.equal(x, y)


@pytest.mark.parametrize("form", ["kappa", "shear", "grad"])
def test_deep_pass_equals_steps(rrp, form):
    """Forty steps through ten periods, launched in groups that hold no more
    than a whole grid's records, against the steps one by one: bit for bit."""
    import torch
    g = synth.Grid((48, 48, 48), 62.4)
    b = synth.Bundle(29, 18, synth.deg(3), synth.deg(2), (31.0, 30.0, 1.0), 9.9 * g.n[2] * g.h)
    cuts = np.linspace(b.chi_s, 0.0, 41)
    steps = [synth.Step(float(x), float(y), 1.0 + 0.01 * i, 0.8) for i, (x, y) in enumerate(zip(cuts[:-1], cuts[1:]))]
    phi = torch.from_numpy(synth.random_field(g.n, 8, np.float32)).cuda()
    tr = rrp.Tracer(b, shear=form == "shear")
    rec = tr.record_buffer(g)
    tr.tidal(g, phi, rec)
    for st in steps:
        tr.step(g, rec, st.chi_a, st.chi_b, st.scale, st.a)
    want = list(tr.finalize()) + (list(tr.shear()) if form == "shear" else [])
    tr.close()
    if form == "grad":
        phi.requires_grad_(True)
        got = list(rrp.TraceKappa.apply(phi, g, b, steps))
    else:
        got = list((rrp.trace_shear if form == "shear" else rrp.trace_kappa)(phi, g, b, steps))[:-1]
    assert len(got) == len(want)
    for x, y in zip(got, want):
        assert torch.equal(x.detach(), y)
