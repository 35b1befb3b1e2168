"""Directions with a component so small that the distance between two crossings
on its axis overflows: the ray crosses nothing on that axis. Against the FP64
oracle (1e-5 of the rms, the map tolerance of the parity tests)."""
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


def _close(got, want):
    got, want = got.cpu().numpy().ravel(), np.asarray(want).ravel()
    assert np.abs(got - want).max() <= TOL * math.sqrt(float(np.mean(want ** 2)))


def _bundle(fov, interp, periodic):
    # (rates of fov / 2 and 0 cells per unit length on the first axis)
    return synth.Bundle(3, 9, fov, synth.deg(9), (15.3, 16.6, 0.4), 70.0, interp=interp, periodic=periodic)


@pytest.mark.parametrize("fov", [1e-37, 4e-39, 1e-39, 1e-42, 1e-300])
@pytest.mark.parametrize("interp", [1, 0])
@pytest.mark.parametrize("periodic", [True, False])
def test_uniform_grid(rrp, oracle_lib, fov, interp, periodic):
    import torch
    g = synth.Grid((32, 34, 90), 32.0)
    b = _bundle(fov, interp, periodic)
    steps = [synth.Step(70.0, 31.0, 1.2, 0.8), synth.Step(31.0, 0.0, 0.9, 1.0)]
    phi = synth.random_field(g.n, 5, np.float32)
    k, kb, _ = rrp.trace_kappa(torch.from_numpy(phi).cuda(), g, b, steps)
    H, d = oracle_lib.fields(g, phi.astype(np.float64))
    o = oracle_lib.trace(b, g, H, d, steps)
    _close(k, o.kappa)
    _close(kb, o.kborn)


@pytest.mark.parametrize("fov", [4e-39, 1e-39])
def test_adaptive_mesh(rrp, oracle_lib, fov):
    import torch
    mesh = synth.amr_random(16, 32.0, 3, 77, threshold=1.05, child_sigma=0.9)
    mesh.phi = [np.asarray(p, np.float32).astype(np.float64)
                for p in synth.amr_sample(mesh, synth.fourier_fn(32.0, 20, 2 * math.pi / 32.0 * 3, 87))]
    b = _bundle(fov, 1, True)
    steps = [synth.Step(45.0, 19.0, 1.1, 0.8), synth.Step(19.0, 0.0, 0.95, 1.0)]
    gm = rrp.AmrMesh(mesh.n, mesh.lmax, mesh.box, mesh.octs, mesh.omega_m)
    flat = np.concatenate([np.asarray(p).reshape(-1) for p in mesh.phi]).astype(np.float32)
    rec = gm.record_buffer()
    gm.tidal(torch.from_numpy(flat).cuda(), rec)
    tr = rrp.Tracer(b)
    for st in steps:
        tr.amr_step(gm, rec, st.chi_a, st.chi_b, st.scale, st.a)
    k, kb = tr.finalize()
    tr.close()
    gm.close()
    o = oracle_lib.amr_trace(b, mesh, steps)
    _close(k, o.kappa)
    _close(kb, o.kborn)
