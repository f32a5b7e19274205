"""A context's first call, on a non-blocking stream, reads tables that were
uploaded for it a moment before: its results are those of a context whose
tables have been there for long."""
import numpy as np
import pytest

from paper_2503_13756_gb300 import swalign

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("projector", ["slice", "splat"])
@pytest.mark.parametrize("metric", ["sw2", "rfsw2"])
def test_first_calls_on_a_non_blocking_stream(projector, metric):
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.rand((4, 96, 96), generator=g, device="cuda")
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    for n in (60, 96, 180, 256, 360, 512):
        p = swalign.make_params(96, n, 32, projector=projector, metric=metric)
        al = swalign.Aligner()
        al.align_batch(x, x[:2], p)
        want = swalign.results_to_numpy(al.align_batch(x, x[:2], p))
        al.close()
        for _ in range(4):
            fresh = swalign.Aligner()
            with torch.cuda.stream(side):
                r = fresh.align_batch(x, x[:2], p)
            side.synchronize()
            assert np.array_equal(swalign.results_to_numpy(r), want)
            fresh.close()
