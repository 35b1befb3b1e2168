"""Steps of many sub-steps of which some cross the periodic seam: the choice per
sub-step (flat offsets inside the grid, wrapped indices across the seam, on one
ray), and the rule by which steps that cross it often take wrapped indices
throughout. The rule is restated here and each case's route asserted, so that a
case cannot come to compare a route with itself. Against the FP64 oracle (1e-5
of the rms, the map tolerance of the parity tests); the two routes bit for bit
in the forms whose passes are, otherwise within that tolerance."""
import math

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

TOL = 1e-5
FORMS = {"default": {}, "shear": {"shear": True}, "method_a": {"method_a": True}, "moments": {"moments": True},
         "generic": {"generic": True}, "plain": {"plain_sums": True}}
KERNELS = ((0.7, -0.011, 0.00004), (-1.3, 0.02, -0.0001))


@pytest.fixture(scope="module")
def rrp():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1601_02012_gb300 import build
    build.build()
    import paper_1601_02012_gb300 as pkg
    return pkg


def _crossings(b, g, st):
    """Seam crossings of the step's extreme rays, and the step's sub-steps."""
    hx = 0.5 * b.fov_x if b.nx > 1 else 0.0
    hy = 0.5 * b.fov_y if b.ny > 1 else 0.0
    ends = [(-math.sin(hx), math.sin(hx)), (-math.sin(hy), math.sin(hy)), (math.cos(math.hypot(hx, hy)), 1.0)]
    total = 0.0
    for a in range(3):
        most = 0.0
        for n in ends[a]:
            x0, x1, side = b.obs[a] + st.chi_a * n, b.obs[a] + st.chi_b * n, g.n[a] * g.h
            x0 += -min(g.h, x0 - x1) if x0 > x1 else min(g.h, x1 - x0)
            most = max(most, abs(math.floor(x0 / side) - math.floor(x1 / side)))
        total += most
    return total, max(1.0, math.ceil((st.chi_a - st.chi_b) / (32.0 * g.h)))


def _heavy(b, g, st):
    crossings, subs = _crossings(b, g, st)
    return 4.0 * crossings > subs


def _trace(rrp, g, b, steps, fields, form, together=False):
    """The maps of the form, and the segment count."""
    import torch
    tr = rrp.Tracer(b, **FORMS[form])
    rec = tr.record_buffer(g)
    if form == "generic":
        tr.set_kernels(KERNELS)
        for c in range(2):
            tr.scalars(g, torch.from_numpy(fields[c]).cuda(), rec, c)
    else:
        tr.tidal(g, torch.from_numpy(fields[0]).cuda(), rec)
    if together:
        tr.steps(g, [rec] * len(steps), steps)
    else:
        for st in steps:
            tr.step(g, rec, st.chi_a, st.chi_b, st.scale, st.a)
    maps = list(tr.finalize()) + (list(tr.shear()) if form == "shear" else [])
    seg = tr.segments()
    tr.close()
    return [m.cpu().numpy() for m in maps], seg


def _close(got, want):
    got, want = got.ravel(), np.asarray(want).ravel()
    assert np.abs(got - want).max() <= TOL * math.sqrt(float(np.mean(want ** 2)))


MIXED = {
    # name: (n, observer in cells, depth in cells, field of view x and y in degrees, step bounds in depths)
    "far_seam": ((64, 60, 120), (30.0, 31.0, 0.5), 205.0, 4.0, 3.0, (1.0, 0.0)),
    "side_and_far": ((48, 70, 250), (3.0, 33.0, 1.0), 416.0, 4.0, 2.0, (1.0, 0.38, 0.0)),
    "sides": ((40, 60, 700), (2.5, 30.0, 20.0), 500.0, 3.0, 9.0, (1.0, 0.0)),
}


@pytest.mark.parametrize("name", sorted(MIXED))
@pytest.mark.parametrize("form", ["default", "shear", "method_a", "moments", "generic"])
def test_mixed_sub_steps_against_oracle(rrp, oracle_lib, name, form):
    n, obs, depth, fx, fy, cuts = MIXED[name]
    h = 1.5
    g = synth.Grid(n, n[0] * h)
    b = synth.Bundle(21, 14, synth.deg(fx), synth.deg(fy), tuple(h * x for x in obs), depth * h)
    steps = [synth.Step(x * b.chi_s, y * b.chi_s, 1.2 - 0.2 * i, 0.8 + 0.1 * i)
             for i, (x, y) in enumerate(zip(cuts[:-1], cuts[1:]))]
    for st in steps:
        crossings, subs = _crossings(b, g, st)
        assert crossings >= 1 and subs >= 5 and not _heavy(b, g, st)
    fields = [synth.random_field(g.n, 77 + c, np.float32) for c in range(2)]
    maps, seg = _trace(rrp, g, b, steps, fields, form)
    if form != "plain" and len(steps) > 1:
        again, seg2 = _trace(rrp, g, b, steps, fields, form, together=True)
        assert seg2 == seg and all(np.array_equal(x, y) for x, y in zip(maps, again))
    phi = fields[0].astype(np.float64)
    if form == "generic":
        want = oracle_lib.trace_kq(b, g, phi, fields[1].astype(np.float64), KERNELS, steps)
    else:
        H, d = oracle_lib.fields(g, phi)
        if form == "method_a":
            kgrad, born = oracle_lib.trace_method_a(b, g, oracle_lib.fields_grad(g, phi), d, steps)
            want = [kgrad + born, born]
        else:
            o = oracle_lib.trace(b, g, H, d, steps)
            assert abs(seg - int(o.nseg.sum())) <= 1e-3 * o.nseg.sum()
            want = [o.kappa, o.kborn] + (list(oracle_lib.trace_shear(b, g, H, steps)) if form == "shear" else [])
    assert len(maps) == len(want)
    for x, y in zip(maps, want):
        _close(x, y)


@pytest.mark.parametrize("name", ["far_seam", "sides"])
@pytest.mark.parametrize("form", sorted(FORMS))
def test_both_routes_agree(rrp, name, form):
    """A bundle so wide that its steps take wrapped indices, and its middle row
    alone, which chooses per sub-step: the shared rays."""
    n, obs, depth, fx, fy, _ = MIXED[name]
    h = 1.5
    g = synth.Grid(n, n[0] * h)
    st = synth.Step(depth * h, 0.0, 1.1, 0.9)
    wide = synth.Bundle(33, 5, synth.deg(fx), synth.deg(70.0), tuple(h * x for x in obs), depth * h)
    narrow = synth.Bundle(33, 1, synth.deg(fx), 0.0, wide.obs, depth * h)
    assert _heavy(wide, g, st) and not _heavy(narrow, g, st) and _crossings(narrow, g, st)[0] >= 1
    fields = [synth.random_field(g.n, 79 + c, np.float32) for c in range(2)]
    a, _ = _trace(rrp, g, wide, [st], fields, form)
    c, _ = _trace(rrp, g, narrow, [st], fields, form)
    for x, y in zip(a, c):
        if form in ("moments", "generic"):
            _close(x[2], y[0])
        else:
            assert np.array_equal(x[2], y[0])
