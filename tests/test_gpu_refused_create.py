"""rr_create while a stream is being captured is refused, and costs no memory:
neither the block it took nor one that the library had kept is lost."""
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


@pytest.mark.parametrize("kept", [True, False])
def test_refused_create_keeps_memory(rrp, kept):
    import torch
    b = synth.Bundle(2048, 2048, 0.1, 0.1, (1.0, 1.0, 0.0), 10.0)   # about 0.2 GB of state
    s = torch.cuda.Stream()

    def refused():
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.stream(s):
            graph.capture_begin()
            try:
                with pytest.raises(rrp.RRError):
                    rrp.Tracer(b)
            finally:
                try:
                    graph.capture_end()
                except RuntimeError:   # (the refused call ended the capture)
                    pass

    rrp.Tracer(b).close()
    rrp.rr_release_cached()
    refused()                      # (what a first capture costs, with nothing kept)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    if kept:
        rrp.Tracer(b).close()
    for _ in range(3):
        refused()
    torch.cuda.synchronize()
    rrp.Tracer(b).close()          # works again
    rrp.rr_release_cached()
    assert torch.cuda.mem_get_info()[0] >= free - (32 << 20)
