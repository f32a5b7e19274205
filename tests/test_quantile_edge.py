"""Trust bound of the quantile kernel's FP32 level counts: a program
(tests/c_abi/quantile_edge.cu) built against the library's internal header
takes every rounding of the count at its worst allowed value (tails of half an
ulp, a fast quotient off by two ulps) around the boundaries between counts, and
no count outside the bound may be wrong.  A bound of 3.4e-7 instead of 4.5e-7
lets through about 1 in 375.  Host code only: no device."""
from tests.test_slice_geometry import _build_and_run


def test_trusted_counts_are_exact(tmp_path):
    assert _build_and_run(tmp_path, "quantile_edge").rstrip().endswith("ok")
