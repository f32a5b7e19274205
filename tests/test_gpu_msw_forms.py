"""Max-sliced W2 tiles at the edges of their forms, against the FP64 oracle: level
counts past one stage of 32 with odd tails (levels staged one by one), and
angle counts just past a multiple of the 64 rows and of the 256 columns of a
tile, up to three column blocks."""
import numpy as np
import pytest

from tests.test_gpu_msw import al, blobs, compare  # noqa: F401  (al: fixture)

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,M", [(72, 33), (144, 35), (270, 65), (600, 37), (540, 34)])
@pytest.mark.parametrize("translation", [1, 0])
def test_msw_tile_edges(al, n, M, translation):  # noqa: F811
    rng = np.random.default_rng(n + M + translation)
    compare(al, blobs(rng, 2, 24), blobs(rng, 3, 24), n=n, M=M, translation=translation)
