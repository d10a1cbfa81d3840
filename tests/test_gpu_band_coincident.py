"""Banded coefficients at samples that nearly coincide: both axes' factors of such a lag are tiny, their
products below the FP64 range, while the Gram entry is 1. With r = 1 the coefficients are the diagonal
FTCG weights. Bar of test_gpu_band (1e-9) against the FP64 pair sums."""
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


@pytest.mark.parametrize("lag", [(1e-170, 1e-170), (1e-300, 3e-20), (5e-324, 1e-310), (1e-99, 1e-99),
                                 (1e-101, 2e-99), (1e-160, 0.0), (1e-12, 1e-200), (1e-7, 3e-6)])
def test_near_coincident_samples(F, lag):
    import torch
    lam = np.concatenate([sasgen.random_case(5, 100, 64, spread=60)[0], [[0.0, 0.0], lag]])
    ref, _ = O.weights_brute(lam, 64)
    with F.Plan(torch.from_numpy(lam).cuda(), 64, 2.0, 6) as p:
        got = p.band(1).cpu().numpy()[:, 0]
    assert np.max(np.abs(got - ref) / ref) < 1e-9
