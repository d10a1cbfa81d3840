"""The forward transform by tiles in shared memory and by the pruned two-pass transform: every
transform length, tile side and layout, narrow and wide windows, ragged last tiles (no power of
two), rasters that wrap, dropped samples, and sample counts on both sides of the rule between the
kernels, against the FP64 oracle. Bar: the FP32 bar of the adjoint's tests (1e-5 rel-L2)."""
import numpy as np
import pytest

import sasgen
from oracle import ftcg_oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    import __graft_entry__ as g
    g.build()
    import paper_1706_08575_gb300 as pkg
    return pkg


@pytest.mark.parametrize("M,N,w,tile,layout,spread,drop", [
    (98304, 128, 8, 32, 2, 128, 0), (98303, 128, 8, 32, 2, 128, 0),      # G = 256, either kernel
    (120000, 256, 6, 64, 2, 300, 5), (110001, 250, 7, 32, 1, 100, 3),    # wraps; ragged, duplicates
    (130000, 90, 13, 64, 1, 90, 0), (100000, 512, 8, 32, 2, 60, 0),
    (100000, 1024, 8, 64, 2, 50, 0), (99000, 2048, 8, 32, 2, 40, 0),
])
def test_forward_against_oracle(F, M, N, w, tile, layout, spread, drop):
    import torch
    lam, _ = sasgen.random_case(M + N, M, N, spread=spread)
    rng = np.random.default_rng(N)
    img = (rng.standard_normal((N, N)) + 1j * rng.standard_normal((N, N))).astype(np.complex64)
    bad = rng.integers(0, M, drop)
    lam[bad] = np.nan
    with F.Plan(torch.from_numpy(lam).cuda(), N, 2.0, w, tile=tile, layout=layout,
                spread_kernel=F.SPREAD_WINDOW, allow_numeric=True) as p:
        out = torch.full((M,), 7.0 + 0j, dtype=torch.complex64, device="cuda")
        got = p.forward(torch.from_numpy(img).cuda(), out).cpu().numpy()
    keep = np.ones(M, bool)
    keep[bad] = False
    ref = O.forward(lam[keep], img.astype(np.complex128), N, 2.0, w)
    assert O.rel_l2(got[keep], ref) < 1e-5
    assert np.all(got[bad] == 0)
