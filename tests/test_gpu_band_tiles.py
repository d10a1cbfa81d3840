"""The banded coefficients at the edges of the kernels' tiles: M around the 32-entry tiles and the
row blocks of the squared band, the smallest and largest r, samples several periods apart. Bar of
test_gpu_band: 1e-9 of the largest coefficient against the oracle's least squares."""
import numpy as np
import pytest

from oracle import ftcg_banded as B
from test_gpu_band import dense_c, dev, lattice

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    import __graft_entry__ as g
    g.build()
    import paper_1706_08575_gb300 as pkg
    return pkg


@pytest.mark.parametrize("M,r", [(1, 1), (31, 2), (32, 12), (33, 3), (65, 1), (97, 6), (257, 5)])
def test_band_at_tile_edges(F, M, r):
    N = 32
    lam, _ = lattice(M, 17, N)
    lam = lam[:M] + N * np.random.default_rng(M).integers(-2, 3, (M, 2))   # several periods
    with F.Plan(dev(lam), N, 2.0, 6) as p:
        got = dense_c(p.band(r).cpu().numpy(), r)
    ref = B.banded_c(B.gram_matrix(lam, N), r)
    assert np.max(np.abs(got - ref)) < 1e-9 * np.max(np.abs(ref))
