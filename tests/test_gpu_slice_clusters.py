"""The Fourier-slice projector's cluster forms: a few images are shared by
clusters of 8, 4 or 2 CTAs each, many take one CTA each.  Every form does the
same arithmetic on each value, so the rows and statuses of an image are the
same bits in a batch of any size, and the one-CTA form is held to the oracle
by the projector's other tests."""
import pytest

from paper_2503_13756_gb300 import swalign

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def al():
    a = swalign.Aligner()
    yield a
    a.close()


# L (odd, even, small, largest of each arrangement), n (one batch of angles,
# part of one, more batches than CTAs); upsampled: images of side L/2
@pytest.mark.parametrize("L,n,up", [
    (5, 4, False), (21, 60, False), (32, 32, False), (64, 360, False), (77, 150, False),
    (96, 128, False), (101, 1024, False), (128, 256, False), (130, 96, False), (160, 256, False),
    (201, 72, False), (256, 360, False), (144, 90, True), (192, 128, True), (256, 1024, True)])
def test_rows_do_not_depend_on_the_batch_size(al, L, n, up):
    import torch
    g = torch.Generator(device="cuda").manual_seed(L * 10 + n)
    side = L // 2 if up else L
    p = swalign.make_params(L, n, 8, projector="slice")
    x = torch.rand((310 if n <= 360 else 160, side, side), generator=g, device="cuda")
    fn = al.project_upsampled if up else al.project
    full = fn(x, p)
    for count in (1, 2, 16, 17, 32, 33, 72, 73, 152):
        for first in (0, x.shape[0] - count):  # the last image too
            rows = fn(x[first:first + count].clone(), p)
            assert torch.equal(rows, full[first:first + count]), (count, first)


@pytest.mark.parametrize("L,q_L", [(64, 64), (160, 160), (256, 128)])
def test_unusable_images_are_found_by_every_cta_of_a_cluster(al, L, q_L):
    """A non-finite pixel anywhere, or no mass, gives status 1 to that query
    alone (the flags of all CTAs meet)."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(L)
    t = torch.rand((2, L, L), generator=g, device="cuda")
    q = torch.rand((6, q_L, q_L), generator=g, device="cuda")
    q[0, 3, 0] = float("nan")
    q[1, q_L - 1, q_L - 1] = float("inf")
    q[2] = 0.0
    q[3] = -1.0
    q[4] = 0.0
    q[4, q_L // 2, q_L - 1] = 1.0  # all mass in one column
    bank = swalign.Bank(al, t, swalign.make_params(L, 64, 16, projector="slice"))
    r = swalign.results_to_numpy(bank.align(q, q_L=q_L, mode=1))
    assert r["status"].tolist() == [1, 1, 1, 1, 0, 0]
    bank.close()
