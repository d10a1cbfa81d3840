"""The rule between the forward transform's two interpolation kernels at the rasters that the average
density does not describe."""
import numpy as np
import pytest

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
