"""A launch that the runtime refuses fails its own call only.  A splat batch of
more than 65,535 images asks for more rows of CTAs than a grid may have: the
host refuses the launch (nothing runs), the call returns SW_ERR_CUDA, and the
calls after it, on the same and on another context, give what they gave
before."""
import numpy as np
import pytest

from paper_2503_13756_gb300 import swalign

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _refused(al, n):
    """n % 4 == 0: the four-view projector; otherwise the tiled one."""
    p = swalign.make_params(2, n, 2)
    with pytest.raises(swalign.SwError) as e:
        al.project(torch.ones((65536, 2, 2), device="cuda"), p)
    assert e.value.status == swalign.SW_ERR_CUDA


def _scales(al):
    x = torch.full((3, 16, 16), 0.5, device="cuda")
    rows, scale = al.project(x, swalign.make_params(16, 8, 4), scale=True)
    return torch.cat([rows.double().flatten(), scale])


def _banded(al):  # two row bands per image (200 < L <= 312)
    x = torch.arange(2 * 210 * 210, device="cuda").reshape(2, 210, 210).float()
    return al.project(x, swalign.make_params(210, 8, 4))


def _max_sliced(al):
    g = torch.Generator(device="cuda").manual_seed(7)
    x = torch.rand((3, 16, 16), generator=g, device="cuda")
    return al.align_batch(x, x[:2].clone(), swalign.make_params(16, 8, 4, metric="msw2"))


def _batch(al):
    g = torch.Generator(device="cuda").manual_seed(8)
    x = torch.rand((3, 16, 16), generator=g, device="cuda")
    return al.align_batch(x, x[:2].clone(), swalign.make_params(16, 8, 4))


@pytest.mark.parametrize("n", [8, 6])
@pytest.mark.parametrize("call", [_scales, _banded, _max_sliced, _batch])
def test_a_refused_launch_does_not_fail_the_next_call(call, n):
    al, other = swalign.Aligner(), swalign.Aligner()
    want = call(al).cpu().numpy()
    for after in (al, other):
        _refused(al, n)
        np.testing.assert_array_equal(call(after).cpu().numpy(), want)
    al.close()
    other.close()
