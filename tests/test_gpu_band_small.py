"""Banded coefficients where a Gram tile is shared by several CTAs (few samples) and where it is not, on
both sides of the line (M = 544 is 153 tile pairs). Bar of test_gpu_band: 1e-9 of the largest coefficient
against the oracle's least squares."""
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


@pytest.mark.parametrize("M,r", [(2, 1), (40, 1), (100, 3), (512, 2), (544, 1), (700, 4)])
def test_band_by_shared_tiles(F, M, r):
    N = 64
    lam, _ = lattice(M, 28, N)
    lam = lam[:M]
    with F.Plan(dev(lam), N, 2.0, 6) as p:
        got = dense_c(p.band(r).cpu().numpy(), r)
    ref = B.banded_c(B.gram_matrix(lam, N), r)
    assert np.max(np.abs(got - ref)) < 1e-9 * np.max(np.abs(ref))
