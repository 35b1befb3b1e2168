"""The adjoint where its warps are ragged: bundles of less than a warp and of
odd sides, rays whose derivative is zero, sub-steps shorter than the forward
walk's (small bundles take those), rays that leave a bounded box, pixels far
apart (many faces per warp) and close together (one): dL/dPhi against the FP64
oracle's gradient, with the tolerances of the gradient tests (1e-5 in l2, 1e-4
of the support's rms at the worst point)."""
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


@pytest.mark.parametrize("nx,ny,fov", [(1, 1, 1.0), (9, 5, 40.0), (33, 7, 0.5), (70, 61, 12.0)])
@pytest.mark.parametrize("interp", [1, 0])
@pytest.mark.parametrize("periodic", [True, False])
@pytest.mark.parametrize("fp64", [False, True])
def test_gradient(rrp, oracle_lib, nx, ny, fov, interp, periodic, fp64):
    import torch
    g = synth.Grid((23, 18, 49), 34.5)
    b = synth.Bundle(nx, ny, synth.deg(fov), synth.deg(0.8 * fov), (16.0, 14.5, 0.7), 110.0, interp=interp,
                     periodic=periodic)
    steps = [synth.Step(110.0, 31.0, 1.2, 0.8), synth.Step(31.0, 0.0, 0.9, 1.0)]
    phi = torch.from_numpy(synth.random_field(g.n, 3, np.float32)).cuda()
    rng = np.random.default_rng(nx + 100 * ny)
    yk, yb = rng.standard_normal((2, ny, nx))
    yk[rng.random((ny, nx)) < 0.3] = 0.0
    yb[yk == 0.0] = 0.0
    if not yk.any():
        yk[:], yb[:] = 1.0, -0.5
    tr = rrp.Tracer(b, fp64_dda=fp64)
    rec = rrp.record_buffer(g)
    tr.tidal(g, phi, rec)
    for st in steps:
        tr.step(g, rec, st.chi_a, st.chi_b, st.scale, st.a)
    tr.finalize()
    got = tr.backward(g, torch.from_numpy(yk).cuda(), torch.from_numpy(yb).cuda()).cpu().numpy()
    tr.close()
    want, _ = oracle_lib.trace_adjoint(b, g, steps, yk.ravel(), yb.ravel())
    support = want != 0
    rms = np.sqrt(np.mean(want[support] ** 2))
    assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)
    assert np.abs(got - want).max() <= 1e-4 * rms


@pytest.mark.parametrize("interp", [1, 0])
def test_nan_stays_with_its_ray(rrp, interp):
    """A NaN and an infinite derivative reach only the points their own rays touch."""
    import torch
    g = synth.Grid((24, 24, 40), 36.0)
    b = synth.Bundle(16, 8, synth.deg(30), synth.deg(20), (18.0, 17.0, 1.0), 50.0, interp=interp)
    st = synth.Step(50.0, 4.0, 1.0, 1.0)
    phi = torch.from_numpy(synth.random_field(g.n, 4, np.float32)).cuda()
    where = rrp.RR_AT_VERTICES if interp else rrp.RR_AT_CENTRES

    def records(y):
        tr = rrp.Tracer(b)
        rec = rrp.record_buffer(g)
        rrp.rr_tidal_tensor(rrp.grid_desc(g), phi, None, rec, where)
        tr.step(g, rec, st.chi_a, st.chi_b, st.scale, st.a)
        tr.finalize()
        out = torch.zeros((g.ncells, 16), dtype=torch.float32, device="cuda")
        rrp.rr_trace_step_adjoint(tr.ctx, 0, torch.from_numpy(y).cuda(), None, out)
        torch.cuda.synchronize()
        tr.close()
        return out.view(torch.float64).cpu().numpy()

    y = np.random.default_rng(1).standard_normal((8, 16))
    clean = records(y)
    bad = [(1, 3, np.nan), (5, 12, np.inf)]
    own = np.zeros(g.ncells, bool)
    for r, c, v in bad:
        one = np.zeros_like(y)
        one[r, c] = 1.0
        own |= (records(one) != 0).any(1)
        y[r, c] = v
    got = records(y)
    assert not np.isfinite(got[own][:, 0]).all()
    rms = np.sqrt(np.mean(clean ** 2))
    assert np.isfinite(got[~own]).all() and np.abs(got[~own] - clean[~own]).max() <= 1e-5 * rms
