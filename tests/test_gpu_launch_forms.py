"""Results do not depend on the form that a batch's size selects, at the sizes
where the launch rules (sw_forms.h) change their choice: every form does the
same arithmetic in the same order for each value, so the results of the same
pairs are the same integers and, up to the order of the FP64 sums over an image
(2^-53 each, amplified by the cancellation in norm + norm - 2 corr, below 1e3
here), the same doubles."""
import numpy as np
import pytest

import oracle
from paper_2503_13756_gb300 import swalign, synth
from tests.parity import level_of, rfsw_level_tol

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


@pytest.mark.parametrize("B", [120, 128])
@pytest.mark.parametrize("n", [4, 36])
def test_ramp_rows_on_each_side_of_the_line(al, B, n):
    """Quantiles of the ramp-filtered parts against the FP64 oracle's, with FFT
    stages taken singly (below 128 bins) and in pairs."""
    L, M = 80, 24
    p = synth.draw_mixtures(np.random.default_rng(B + n), 3, L, ncomp=(2, 5))
    imgs = np.ascontiguousarray(synth.render(p, L), dtype=np.float32)
    par = swalign.make_params(L, n, M, n_bins=B, metric="rfsw2")
    Q = al.quantiles(al.project(imgs, par), par)[0].cpu().numpy()
    z = (np.arange(M) + 0.5) / M
    for i in range(len(imgs)):
        F, _ = oracle.prepare(imgs[i].astype(np.float64))
        U = oracle.project(F, n, B)
        Ut, parts = oracle.ramp_filter(U), oracle.rfsw_parts(U)
        for part in range(2):
            for k in range(n):
                lev = level_of(Q[i, part, k].astype(np.float64), parts[part][k], 2.0 / L)
                assert np.abs(lev - z).max() <= rfsw_level_tol(Ut[k], parts[part][k]), (i, part, k)


@pytest.mark.parametrize("nt,counts", [(129, (216, 217)), (300, (302, 303))])
def test_best_template_on_each_side_of_the_line(al, nt, counts):
    """A block or a warp per query: the least d2 of the usable results, the
    lowest index on ties (every third template is a copy of the first)."""
    g = torch.Generator(device="cuda").manual_seed(nt)
    p = swalign.make_params(8, 8, 4)
    t = torch.rand((nt, 8, 8), generator=g, device="cuda")
    t[::3] = t[0]
    t[1] = 0.0
    q = torch.cat([t[:3], torch.rand((counts[-1] - 3, 8, 8), generator=g, device="cuda")])
    every = swalign.results_to_numpy(al.align_batch(q, t, p)).reshape(-1, nt)
    j = np.where(every["status"] == 0, every["d2"], np.inf).argmin(1)
    for count in counts:
        best = swalign.results_to_numpy(al.align_batch(q[:count].clone(), t, p, mode=1))
        use = best["status"] == 0
        assert np.array_equal(use, every["status"][:count].min(1) == 0)
        assert np.array_equal(best["template_index"][use], j[:count][use])
        assert np.array_equal(best["d2"][use], every["d2"][np.arange(count), j[:count]][use])
