"""Results do not depend on how many images share a call: a few images go
through the cluster forms of the kernels (several CTAs per image), many
through one CTA each, with the same operations and the same order of every
FP32 sum, so the results of the same pairs are the same integers and, up to
the order of the FP64 sums over an image (2^-53 each, amplified by the
cancellation in norm + norm - 2 corr, below 1e3 here), the same doubles."""
import numpy as np
import pytest

from paper_2503_13756_gb300 import swalign

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def al():
    a = swalign.Aligner()
    yield a
    a.close()


# angle counts of every spectrum form (two and one CTA per SM, n > 512, all
# pairs of FFT stages), level counts at the edges of the 32-level batches,
# one and two parts
@pytest.mark.parametrize("n,M,metric", [
    (4, 1, "sw2"), (64, 33, "sw2"), (90, 256, "sw2"), (120, 128, "rfsw2"), (180, 101, "sw2"),
    (200, 160, "sw2"), (256, 128, "sw2"), (256, 129, "rfsw2"), (360, 256, "sw2"),
    (384, 97, "sw2"), (480, 256, "sw2"), (500, 129, "rfsw2"), (512, 257, "sw2"),
    (720, 64, "sw2"), (1024, 100, "sw2")])
@pytest.mark.parametrize("precision", ["fp32", "bf16", "fp32_simt"])
def test_pairs_do_not_depend_on_the_batch(al, n, M, metric, precision):
    import torch
    g = torch.Generator(device="cuda").manual_seed(n + M)
    p = swalign.make_params(32, n, M, precision=precision, metric=metric)
    q = torch.rand((420, 32, 32), generator=g, device="cuda")
    t = torch.rand((2, 32, 32), generator=g, device="cuda")
    full = swalign.results_to_numpy(al.align_batch(q, t, p)).reshape(-1, 2)
    for count in (1, 6, 30, 70, 130):
        r = swalign.results_to_numpy(al.align_batch(q[:count].clone(), t, p)).reshape(-1, 2)
        for f in ("best_l", "status", "template_index"):
            assert np.array_equal(r[f], full[f][:count]), (count, f)
        for f in ("shift", "d2"):
            assert np.allclose(r[f], full[f][:count], rtol=1e-12, atol=1e-14), (count, f)


@pytest.mark.parametrize("nt", [1, 31, 128, 129, 300, 1025])
def test_best_template_is_the_argmin_of_all_pairs(al, nt):
    """Mode 1 (a warp per query up to 128 templates, a block above) picks the
    least d2, the lowest index on ties, of the usable results of mode 0; the
    first, a middle and the last template are copies, and one is unusable."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(nt)
    p = swalign.make_params(16, 8, 4)
    t = torch.rand((nt, 16, 16), generator=g, device="cuda")
    t[nt // 2] = t[0]
    t[-1] = t[0]
    if nt > 2:
        t[1] = 0.0
    q = torch.cat([t[:1], torch.rand((9, 16, 16), generator=g, device="cuda")])
    every = swalign.results_to_numpy(al.align_batch(q, t, p)).reshape(-1, nt)
    best = swalign.results_to_numpy(al.align_batch(q, t, p, mode=1))
    d = np.where(every["status"] == 0, every["d2"], np.inf)
    j = d.argmin(1)
    assert np.array_equal(best["template_index"], j)
    assert np.array_equal(best["d2"], d[np.arange(len(j)), j])
    assert np.array_equal(best["best_l"], every["best_l"][np.arange(len(j)), j])
