"""The shared-memory transforms of the smallest grid sides (64 and 128): adjoint, forward and batch
against the FP64 oracle, with rasters that fill and that wrap the grid. Bar: that of test_gpu_parity (1e-5 rel-L2, more where the window division amplifies)."""
import numpy as np
import pytest

import sasgen
from oracle import ftcg_oracle as O
from test_gpu_parity import image_tol

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    import __graft_entry__ as g
    g.build()
    import paper_1706_08575_gb300 as pkg
    return pkg


@pytest.mark.parametrize("N,sigma,w,spread", [(32, 2.0, 8, 10), (32, 2.0, 6, 40), (64, 2.0, 7, 200),
                                              (64, 1.0, 4, 30), (100, 1.28, 8, 60), (50, 1.28, 5, 20)])
def test_small_sides(F, N, sigma, w, spread):
    import torch
    lam, v = sasgen.random_case(N + w, 700, N, sigma, w, spread)
    v = v.astype(np.complex64)
    rng = np.random.default_rng(w)
    img = (rng.standard_normal((N, N)) + 1j * rng.standard_normal((N, N))).astype(np.complex64)
    lt, vt = torch.from_numpy(lam).cuda(), torch.from_numpy(v).cuda()
    with F.Plan(lt, N, sigma, w) as p:
        assert p.G in (64, 128)
        a = p.adjoint(vt).cpu().numpy()
        f = p.forward(torch.from_numpy(img).cuda()).cpu().numpy()
        a2 = p.adjoint(vt).cpu().numpy()           # the grid held the forward's cells in between
    with F.Batch([lt, lt[:300].contiguous()], [N, N], sigma, w) as b:
        bi = b.adjoint([vt, vt[:300].contiguous()])
        bi = [x.cpu().numpy() for x in bi]
    ref = O.adjoint(lam, v.astype(np.complex128), N, sigma, w)
    bar = image_tol(N, sigma, w)
    assert O.rel_l2(a, ref) < bar and O.rel_l2(a2, ref) < bar
    assert O.rel_l2(f, O.forward(lam, img.astype(np.complex128), N, sigma, w)) < bar
    assert O.rel_l2(bi[0], ref) < bar
    assert O.rel_l2(bi[1], O.adjoint(lam[:300], v[:300].astype(np.complex128), N, sigma, w)) < bar
