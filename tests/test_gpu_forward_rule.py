"""The rule between the forward transform's two interpolation kernels at the rasters that the average
density does not describe."""
import numpy as np
import pytest

from oracle import ftcg_oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    import __graft_entry__ as g
    g.build()
    import paper_1706_08575_gb300 as pkg
    return pkg


@pytest.mark.parametrize("M,N,tile,layout", [(98304, 64, 32, 2), (98303, 64, 32, 2), (100001, 50, 64, 1)])
def test_all_samples_dropped(F, M, N, tile, layout):
    """Samples without a finite coordinate read zero, also when there are no others."""
    import torch
    lam = torch.full((M, 2), float("nan"), dtype=torch.float64, device="cuda")
    img = torch.ones((N, N), dtype=torch.complex64, device="cuda")
    with F.Plan(lam, N, 2.0, 8, tile=tile, layout=layout, allow_numeric=True) as p:
        out = torch.full((M,), 7.0 + 0j, dtype=torch.complex64, device="cuda")
        assert np.all(p.forward(img, out).cpu().numpy() == 0)
        x, hist, done = p.cgls(torch.ones(M, dtype=torch.complex64, device="cuda"), iters=2)
        assert np.all(x.cpu().numpy() == 0) and np.all(hist == 0) and done == 0


@pytest.mark.parametrize("frac", [0.3, 0.5, 0.97])
@pytest.mark.parametrize("tile,layout", [(32, 2), (64, 1)])
def test_uneven_rasters(F, frac, tile, layout):
    """A share of the samples in one spot, on both sides of the limit on CTAs without samples. Bar: the
    FP32 bar of the adjoint's tests."""
    import torch
    M, N = 120000, 128
    rng = np.random.default_rng(7)
    spot = int(M * frac)
    lam = np.concatenate([rng.random((spot, 2)) * 3.0, (rng.random((M - spot, 2)) - 0.5) * N])
    lam = lam[rng.permutation(M)]
    img = (rng.standard_normal((N, N)) + 1j * rng.standard_normal((N, N))).astype(np.complex64)
    with F.Plan(torch.from_numpy(lam).cuda(), N, 2.0, 8, tile=tile, layout=layout) as p:
        got = p.forward(torch.from_numpy(img).cuda()).cpu().numpy()
    assert O.rel_l2(got, O.forward(lam, img.astype(np.complex128), N, 2.0, 8)) < 1e-5


@pytest.mark.parametrize("M,N,w,tile,drop", [
    (262144, 90, 16, 64, 0), (262143, 90, 16, 64, 2), (270001, 100, 13, 32, 3),      # wide windows
    (120000, 128, 8, 64, 0), (120000, 250, 8, 64, 4), (120000, 250, 5, 32, 0), (100000, 128, 12, 64, 1),
])
def test_duplicate_layout(F, M, N, w, tile, drop):
    """Every sample written once by the tile of its first tap, dropped ones read zero, on both sides of
    the duplicate layout's lines. Bar: the FP32 bar of the adjoint's tests."""
    import torch
    rng = np.random.default_rng(M + N)
    lam = (rng.random((M, 2)) - 0.5) * N
    img = (rng.standard_normal((N, N)) + 1j * rng.standard_normal((N, N))).astype(np.complex64)
    bad = rng.choice(M, drop, replace=False)
    lam[bad] = np.inf
    with F.Plan(torch.from_numpy(lam).cuda(), N, 2.0, w, tile=tile, layout=1, allow_numeric=True) as p:
        out = torch.full((M,), 7.0 + 0j, dtype=torch.complex64, device="cuda")
        got = p.forward(torch.from_numpy(img).cuda(), out).cpu().numpy()
    keep = np.ones(M, bool)
    keep[bad] = False
    assert O.rel_l2(got[keep], O.forward(lam[keep], img.astype(np.complex128), N, 2.0, w)) < 1e-5
    assert np.all(got[bad] == 0)
