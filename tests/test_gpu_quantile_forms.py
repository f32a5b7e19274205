"""Quantile kernel on the GPU at the edges of its forms: bin counts around
multiples of 32 and past the register form (B > 384), level counts around the
groups of 64 and 128, both level rules, and levels that fall exactly on nodes
of the CDF beside empty bins (Eq. inv_cdf with the ">=" of App. A.1.1)."""
import numpy as np
import pytest

from paper_2503_13756_gb300 import swalign

pytestmark = pytest.mark.gpu

# (L, n_bins): n_bins even and >= the default bin count of L
BINS = [(2, 4), (16, 32), (17, 34), (40, 62), (40, 64), (60, 96), (100, 158), (128, 192),
        (200, 320), (240, 350), (256, 384), (256, 386), (300, 512), (512, 2048)]
LEVELS = [1, 2, 63, 64, 65, 127, 128, 129, 256, 1024]


@pytest.fixture(scope="module")
def al():
    a = swalign.Aligner()
    yield a
    a.close()


@pytest.mark.parametrize("rule", [0, 1])
@pytest.mark.parametrize("L,B", BINS)
def test_register_forms_match_the_run_time_form(al, L, B, rule):
    """The same rows in the middle of rows of more than 384 bins, the rest
    empty, take the run-time form.  Its partial sums run in another order, so
    tau - F differs by at most 2^-46 F_B: a rounding of the numerator.  With
    the fast quotient (2 ulp in either form, ulp <= 2^-23 of the fraction)
    the fractions differ by at most 5 ulp and Q = e_j + h frac by that times h
    and two roundings of Q."""
    rng = np.random.default_rng(B + rule)
    pad = max(0, (400 - B) // 2)
    big = B + 2 * pad
    h = 2.0 / L
    for M in LEVELS if B <= 512 else (64, 129):
        U = rng.uniform(0.5, 1.0, size=(2, 4, B)).astype(np.float32)
        W = np.zeros((2, 4, big), dtype=np.float32)
        W[..., pad:pad + B] = U
        q, w = (al.quantiles(x, swalign.make_params(L, 4, M, n_bins=x.shape[-1], level_rule=rule))
                [0].cpu().numpy().astype(np.float64) for x in (U, W))
        if rule:  # tau = 0 is the domain's left end, which the padding moves
            assert np.all(q[..., 0] == np.float32(-0.5 * B * np.float32(h)))
            q, w = q[..., 1:], w[..., 1:]
        tol = 5 * 2.0 ** -23 * h + 2 * 2.0 ** -24 * np.abs(w)
        assert np.all(np.abs(q - w) <= tol), (M, np.abs(q - w).max())


@pytest.mark.parametrize("scale", [1.0, 2.0 ** -120, 2.0 ** 90])
@pytest.mark.parametrize("L,B", [(17, 34), (128, 192), (256, 384), (300, 512)])
def test_levels_on_nodes_take_the_left_end(al, L, B, scale):
    """K unit masses in alternate bins and levels p / K: every level is a node
    of the CDF, and the quantile is the right end of bin 2 (p - 1), the left
    end of the empty bin after it, for every mass scale (all sums exact)."""
    K = B // 2
    U = np.zeros((1, 4, B), dtype=np.float32)
    U[..., ::2] = scale
    p = swalign.make_params(L, 4, K, n_bins=B, level_rule=1)
    q = al.quantiles(U, p)[0].cpu().numpy()[0, 0].astype(np.float64)
    h = 2.0 / L
    lev = np.arange(K)
    want = np.where(lev == 0, -0.5 * B * h, (2 * (lev - 1) + 1 - B / 2) * h)
    assert np.all(np.abs(q - want) <= 2.5e-7 * np.abs(want) + 1e-7)
