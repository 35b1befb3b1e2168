"""Per-sub-step choice of the record addressing (whole-grid records): sub-steps
that lie inside the grid without a wrap take 32-bit point offsets, the others
wrapped vertex indices. Cones of many sub-steps that mix both, that end exactly
on the box face and that a bounded box clips, for every form: against the FP64
oracle (1e-5 of the rms, the map tolerance of the parity tests), and single
steps on whole-grid records bit for bit against box-local ones."""
import math

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

TOL = 1e-5


@pytest.fixture(scope="module")
def rrp():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1601_02012_gb300 import build
    build.build()
    import paper_1601_02012_gb300 as pkg
    return pkg


CASES = {
    # name: (n, observer in cells, periodic, chi_s in cells, field of view)
    "face": ((70, 66, 130), (35.0, 33.0, 0.0), True, 130.0, 12.0),         # every sub-step inside, ends on z = 0
    "through_seams": ((40, 36, 90), (20.3, 17.6, 0.0), True, 250.0, 40.0),   # inside and across, several periods
    "corner": ((64, 64, 64), (0.0, 0.0, 0.0), True, 64.0, 15.0),           # rays on both sides of two seams
    "small_grid": ((9, 8, 7), (4.5, 4.0, 0.0), True, 80.0, 10.0),          # sub-steps longer than the box
    "bounded": ((60, 44, 100), (30.0, 22.0, 0.0), False, 100.0, 50.0),     # sides and far face clip the rays
    "bounded_outside": ((50, 50, 50), (25.5, 20.0, -60.0), False, 200.0, 30.0),
}


def _setup(name):
    n, obs, periodic, chi_s, fov = CASES[name]
    h = 1.5
    g = synth.Grid(n, n[0] * h)
    b = synth.Bundle(21, 14, synth.deg(fov), synth.deg(0.7 * fov), tuple(h * x for x in obs), chi_s * h,
                     periodic=periodic)
    cs = b.chi_s
    return g, b, [synth.Step(cs, 0.41 * cs, 1.2, 0.8), synth.Step(0.41 * cs, 0.0, 0.9, 1.0)]


def _close(got, want):
    got, want = np.asarray(got.cpu()).ravel(), np.asarray(want).ravel()
    rms = math.sqrt(float(np.mean(want ** 2)))
    assert np.abs(got - want).max() <= TOL * rms


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("form", ["default", "shear", "method_a"])
@pytest.mark.parametrize("interp", [1, 0])
def test_against_oracle(rrp, oracle_lib, name, form, interp):
    import torch
    g, b, steps = _setup(name)
    b.interp = interp
    phi = synth.random_field(g.n, 77, np.float32)
    H, d = oracle_lib.fields(g, phi.astype(np.float64))
    ph = torch.from_numpy(phi).cuda()
    tr = rrp.Tracer(b, shear=form == "shear", method_a=form == "method_a")
    rec = tr.record_buffer(g)
    tr.tidal(g, ph, rec)
    for st in steps:
        tr.step(g, rec, st.chi_a, st.chi_b, st.scale, st.a)
    k, kb = tr.finalize()
    if form == "method_a":
        kgrad, born = oracle_lib.trace_method_a(b, g, oracle_lib.fields_grad(g, phi.astype(np.float64)), d, steps)
        _close(k, kgrad + born)
        _close(kb, born)
    else:
        o = oracle_lib.trace(b, g, H, d, steps)
        assert abs(tr.segments() - int(o.nseg.sum())) <= 1e-3 * o.nseg.sum()
        _close(k, o.kappa)
        _close(kb, o.kborn)
        if form == "shear":
            for got, want in zip(tr.shear(), oracle_lib.trace_shear(b, g, H, steps)):
                _close(got, want)
    tr.close()


def test_whole_grid_equals_box_local(rrp):
    import torch
    g, b, _ = _setup("face")
    cs = b.chi_s
    edges = [cs, 0.6 * cs, 0.3 * cs, 0.05 * cs, 0.0]
    steps = [synth.Step(x, y, 1.1, 0.9) for x, y in zip(edges[:-1], edges[1:])]
    ph = torch.from_numpy(synth.random_field(g.n, 78, np.float32)).cuda()
    out = []
    for boxed in (False, True):
        tr = rrp.Tracer(b)
        if boxed:
            boxes = [tr.footprint(g, st.chi_a, st.chi_b, pad=1) for st in steps]
            recs = [tr.tidal_box(g, ph, rrp.box_record_buffer(bb), bb) for bb in boxes]
            tr.steps(g, recs, steps, boxes=boxes)
        else:
            rec = rrp.record_buffer(g)
            tr.tidal(g, ph, rec)
            for st in steps:
                tr.step(g, rec, st.chi_a, st.chi_b, st.scale, st.a)
        out.append([m.cpu().numpy() for m in tr.finalize()] + [tr.segments()])
        tr.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    assert out[0][2] == out[1][2]


@pytest.mark.parametrize("form", ["default", "shear", "method_a", "plain"])
@pytest.mark.parametrize("name", ["through_seams", "small_grid", "corner"])
def test_wrapped_equals_per_sub_step(rrp, name, form):
    """The same ray segments by wrapped indices throughout (a bundle whose field
    of view makes it cross the seam often) and per sub-step (its narrow middle
    row alone, which does not): the shared rays bit for bit."""
    import torch
    g, b, _ = _setup(name)
    st = synth.Step(b.chi_s, 0.0, 1.1, 0.9)
    ph = torch.from_numpy(synth.random_field(g.n, 79, np.float32)).cuda()
    out = []
    for fov in (b.fov_y, 0.0):
        # odd row count: the middle row lies at angle zero on this axis in both
        c = synth.Bundle(b.nx, 5 if fov else 1, b.fov_x, fov, b.obs, b.chi_s)
        tr = rrp.Tracer(c, shear=form == "shear", method_a=form == "method_a", plain_sums=form == "plain")
        rec = tr.record_buffer(g)
        tr.tidal(g, ph, rec)
        tr.step(g, rec, st.chi_a, st.chi_b, st.scale, st.a)
        maps = list(tr.finalize()) + (list(tr.shear()) if form == "shear" else [])
        out.append([m[m.shape[0] // 2].cpu().numpy() for m in maps])
        tr.close()
    for x, y in zip(*out):
        assert np.array_equal(x, y)
