"""The adjoint on a grid of more than 2^32 points, whose point numbers need 64
bits: the last planes of a 4096 x 1025 x 1024 grid against the same rays in a
grid of 16 planes, with the l2 tolerance of the gradient tests (1e-5). The
records of the large grid (275 GB) are not allocated: a bundle touches the
planes of its footprint only, so the buffers hold these planes and their
addresses are given as those of the grid's first point."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

N1, N2, LAST = 1025, 1024, 4096   # plane: 1 049 600 points; 4096 of them: 2^32 + 4 194 304 points
KEPT = 9                          # planes in the buffers
DEPTH = 60.0


@pytest.fixture(scope="module")
def rrp():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1601_02012_gb300 import build
    build.build()
    import paper_1601_02012_gb300 as pkg
    return pkg


def _grid_and_bundle(planes, interp):
    g = synth.Grid((planes, N1, N2), float(planes))
    return g, synth.Bundle(13, 9, synth.deg(4), synth.deg(3), (planes - 4.1, 512.3, 0.7), DEPTH, interp=interp)


@pytest.mark.parametrize("interp", [1, 0])
@pytest.mark.parametrize("fp64", [False, True])
def test_points_past_32_bits(rrp, interp, fp64):
    import torch
    plane = N1 * N2
    assert LAST * plane > 2 ** 32 > (LAST - KEPT) * plane
    y = torch.from_numpy(np.random.default_rng(4).standard_normal((2, 9, 13))).cuda()
    grads = []
    for planes in (16, LAST):
        g, b = _grid_and_bundle(planes, interp)
        tr = rrp.Tracer(b, fp64_dda=fp64)
        box = tr.footprint(g, DEPTH, 0.0)
        first = planes - KEPT
        # every point the step touches lies in the planes that the buffers hold
        assert first <= box[0] and box[1] <= planes
        rec = torch.zeros((KEPT * plane, 8), dtype=torch.float32, device="cuda")
        grad = torch.zeros((KEPT * plane, 16), dtype=torch.float32, device="cuda")
        tr.step(g, rec.data_ptr() - 32 * first * plane, DEPTH, 0.0, 1.1, 0.9)
        rrp.rr_trace_step_adjoint(tr.ctx, 0, y[0].contiguous(), y[1].contiguous(), grad.data_ptr() - 64 * first * plane)
        tr.finalize()
        tr.close()
        grads.append(grad.view(torch.float64))
    want, got = grads
    assert float(want.abs().max()) > 0
    assert float((got - want).norm()) <= 1e-5 * float(want.norm())
