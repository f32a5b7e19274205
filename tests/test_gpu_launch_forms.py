"""Results do not depend on the form that a batch's size selects, at the sizes
where the launch rules (sw_forms.h) change their choice: every form does the
same arithmetic in the same order for each value, so the results of the same
pairs are the same integers and, up to the order of the FP64 sums over an image
(2^-53 each, amplified by the cancellation in norm + norm - 2 corr, below 1e3
here), the same doubles."""
import numpy as np
import pytest

from paper_2503_13756_gb300 import swalign

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def al():
    a = swalign.Aligner()
    yield a
    a.close()


def _check(al, n, M, counts, total, **kw):
    g = torch.Generator(device="cuda").manual_seed(n * 7 + M)
    p = swalign.make_params(16, n, M, **kw)
    q = torch.rand((total, 16, 16), generator=g, device="cuda")
    t = torch.rand((2, 16, 16), generator=g, device="cuda")
    full = swalign.results_to_numpy(al.align_batch(q, t, p)).reshape(-1, 2)
    assert np.all(full["status"] == 0)
    for count in counts:
        r = swalign.results_to_numpy(al.align_batch(q[:count].clone(), t, p)).reshape(-1, 2)
        for f in ("best_l", "status", "template_index"):
            assert np.array_equal(r[f], full[f][:count]), (count, f)
        for f in ("shift", "d2"):
            assert np.allclose(r[f], full[f][:count], rtol=1e-12, atol=1e-14), (count, f)


# spectra in clusters of every width 2..8 (two images more than the count),
# with one and several batches per CTA, even and odd level counts, one and
# two parts, at the last count of a width and the first of the next
@pytest.mark.parametrize("n,M,kw", [
    (256, 128, {}), (360, 256, {}), (360, 160, {"precision": "bf16"}), (240, 223, {}),
    (120, 96, {"metric": "rfsw2"}), (512, 321, {"precision": "fp32_simt"}), (720, 100, {}),
    (64, 1024, {})])
def test_spectrum_clusters_of_every_width(al, n, M, kw):
    _check(al, n, M, (1, 13, 14, 21, 22, 26, 27, 34, 35, 44, 45, 56, 72, 73, 95, 96, 150), 320, **kw)


# many images: plain and half batches on each side of the rule's lines
@pytest.mark.parametrize("n,M,kw", [
    (360, 100, {}), (360, 64, {"precision": "bf16"}), (320, 9, {}), (512, 129, {}),
    (64, 129, {}), (200, 96, {"metric": "rfsw2"}), (8, 256, {"precision": "bf16"}),
    (720, 64, {}), (900, 101, {"precision": "fp32_simt"}), (1000, 20, {"metric": "rfsw2"})])
def test_spectra_of_many_images(al, n, M, kw):
    _check(al, n, M, (150, 153, 303, 309, 455, 470, 599), 640, **kw)
