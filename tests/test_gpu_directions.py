"""Ray directions: one thread computes a quarter bundle's angles and writes the
four mirrored rays. Sides of one ray, odd and even sides, bands that hold one
of two mirrored rows, both or neither: maps against the FP64 oracle (1e-5 of
the rms: the map tolerance of the parity tests) and bands bit for bit against
the whole bundle."""
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


@pytest.mark.parametrize("nx,ny,bands", [(1, 1, [0, 1]), (1, 4, [0, 1, 4]), (2, 1, [0, 1]), (7, 9, [0, 2, 4, 5, 9]),
                                         (34, 6, [0, 1, 6]), (33, 18, [0, 8, 16, 18])])
def test_quarters_and_bands(rrp, oracle_lib, nx, ny, bands):
    import torch
    g = synth.Grid((20, 24, 28), 40.0)
    b = synth.Bundle(nx, ny, synth.deg(14), synth.deg(9), (19.0, 25.0, 3.0), 50.0)
    st = synth.Step(50.0, 2.0, 1.1, 0.9)
    phi = synth.random_field(g.n, 31, np.float32)
    rec = rrp.record_buffer(g)
    rrp.rr_tidal_tensor(rrp.grid_desc(g), torch.from_numpy(phi).cuda(), None, rec)

    def trace(rows=None):
        tr = rrp.Tracer(b, rows=rows)
        tr.step(g, rec, st.chi_a, st.chi_b, st.scale, st.a)
        out = [m.cpu().numpy() for m in tr.finalize()]
        tr.close()
        return out

    whole = trace()
    parts = [trace((y0, y1)) for y0, y1 in zip(bands[:-1], bands[1:])]
    for i in range(2):
        assert np.array_equal(np.concatenate([p[i] for p in parts]), whole[i])
    H, d = oracle_lib.fields(g, phi.astype(np.float64))
    o = oracle_lib.trace(b, g, H, d, [st])
    for got, want in zip(whole, (o.kappa, o.kborn)):
        assert np.abs(got.ravel() - want).max() <= 1e-5 * np.sqrt(np.mean(want ** 2))
