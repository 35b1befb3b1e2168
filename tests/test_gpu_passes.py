"""Passes on one potential (trace_kappa, trace_shear, trace_method_a,
trace_tiles, TraceKappa): one record buffer for all steps and many steps per
launch, against the steps one by one on their own records, bit for bit; for
cones whose footprints share a box, have boxes of their own, reach around the
box, or leave a bounded one."""
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


def _bundle(where, interp, periodic):
    n = (36, 44, 70)
    h = 1.3
    g = synth.Grid(n, n[0] * h)
    obs, chi = {"inside": ((18.0, 22.0, 3.0), 60.0), "face": ((18.0, 22.0, 0.0), 70.0),
                "around": ((1.0, 43.0, 20.0), 160.0)}[where]
    b = synth.Bundle(37, 22, synth.deg(11), synth.deg(8), tuple(h * x for x in obs), chi * h, interp=interp,
                     periodic=periodic)
    cuts = np.linspace(1.0, 0.0, 20) ** 1.3 * b.chi_s
    cuts[0], cuts[-1] = b.chi_s, 0.0
    steps = [synth.Step(float(x), float(y), 1.0 + 0.01 * i, 0.8 + 0.01 * i)
             for i, (x, y) in enumerate(zip(cuts[:-1], cuts[1:]))]
    return g, b, steps


def _one_by_one(rrp, g, b, steps, phi, footprint, tiles=None, **form):
    tr = rrp.Tracer(b, **form)
    for obs in tiles or [None]:
        if obs is not None:
            tr.set_observer(obs)
        rec = tr.record_buffer(g)
        for st in steps:
            tr.tidal(g, phi, rec, bbox=tr.footprint(g, st.chi_a, st.chi_b) if footprint else None)
            tr.step(g, rec, st.chi_a, st.chi_b, st.scale, st.a)
    out = list(tr.finalize())
    seg = tr.segments()
    if form.get("shear"):
        out += list(tr.shear())
    tr.close()
    return [m.cpu().numpy() for m in out], seg


@pytest.mark.parametrize("where", ["inside", "face", "around"])
@pytest.mark.parametrize("own_boxes", [False, True])
@pytest.mark.parametrize("form", ["kappa", "ngp", "fp64", "shear", "method_a", "method_a_ngp", "bounded", "whole"])
def test_pass_equals_steps(rrp, monkeypatch, where, own_boxes, form):
    import torch
    interp = 0 if form.endswith("ngp") else 1
    g, b, steps = _bundle(where, interp, form != "bounded")
    phi = torch.from_numpy(synth.random_field(g.n, 5, np.float32)).cuda()
    if own_boxes:
        monkeypatch.setattr(rrp, "_LAUNCH_POINTS", -10 ** 9)
    kw = {"shear": {"shear": True}, "method_a": {"method_a": True}, "method_a_ngp": {"method_a": True},
          "fp64": {"fp64_dda": True}}.get(form, {})
    want, seg = _one_by_one(rrp, g, b, steps, phi, form != "whole", **kw)
    if form == "shear":
        got = rrp.trace_shear(phi, g, b, steps)
    elif form.startswith("method_a"):
        got = rrp.trace_method_a(phi, g, b, steps)
    else:
        got = rrp.trace_kappa(phi, g, b, steps, fp64_dda=form == "fp64", footprint=form != "whole")
    assert got[-1] == seg
    for x, y in zip(got[:-1], want):
        assert np.array_equal(x.cpu().numpy(), y)


def test_tiles_equal_steps(rrp):
    import torch
    g, b, steps = _bundle("face", 1, False)
    b.chi_s *= 2.2
    steps = [synth.Step(2.2 * s.chi_a, 2.2 * s.chi_b, s.scale, s.a) for s in steps]
    phi = torch.from_numpy(synth.random_field(g.n, 6, np.float32)).cuda()
    depth = g.n[2] * g.h
    tiles = [(b.obs[0], b.obs[1], -i * depth) for i in range(3)]
    want, seg = _one_by_one(rrp, g, b, steps, phi, True, tiles)
    got = rrp.trace_tiles([(phi, g, o) for o in tiles], b, steps)
    assert got[2] == seg
    for x, y in zip(got[:2], want):
        assert np.array_equal(x.cpu().numpy(), y)


def test_contexts_reuse_memory(rrp):
    """Contexts of several forms and sizes made and closed in turn, and in four
    threads with a stream each: every one starts from zeros; the memory kept
    for later ones goes back on request."""
    import threading

    import torch
    g, b, steps = _bundle("face", 1, True)
    phi = torch.from_numpy(synth.random_field(g.n, 7, np.float32)).cuda()
    small = synth.Bundle(9, 7, b.fov_x, b.fov_y, b.obs, b.chi_s)
    first = [[m.cpu().numpy() for m in rrp.trace_kappa(phi, g, c, steps)[:2]] for c in (b, small)]
    shear = [m.cpu().numpy() for m in rrp.trace_shear(phi, g, b, steps)[:4]]
    bad = []

    def work(seed):
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.default_stream())
        with torch.cuda.stream(s):
            for i in range(6):
                c = (b, small)[(seed + i) % 2]
                got = rrp.trace_kappa(phi, g, c, steps, stream=s)
                for x, y in zip(got[:2], first[(seed + i) % 2]):
                    if not np.array_equal(x.cpu().numpy(), y):
                        bad.append((seed, i))
                got = rrp.trace_shear(phi, g, b, steps, stream=s)
                for x, y in zip(got[:4], shear):
                    if not np.array_equal(x.cpu().numpy(), y):
                        bad.append((seed, i, "shear"))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
    big = synth.Bundle(2048, 2048, b.fov_x, b.fov_y, b.obs, b.chi_s)   # about 0.2 GB of state
    rrp.Tracer(big).close()
    torch.cuda.synchronize()
    kept = torch.cuda.mem_get_info()[0]
    rrp.rr_release_cached()
    assert torch.cuda.mem_get_info()[0] >= kept + (100 << 20)
