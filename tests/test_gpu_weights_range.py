"""Exact weights of rasters that the usual ones do not describe: far from the origin, strongly uneven,
window widths and oversamplings whose lag grid is no power of two."""
import numpy as np
import pytest

import sasgen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    import __graft_entry__ as g
    g.build()
    import paper_1706_08575_gb300 as pkg
    return pkg


def weights(F, lam, N, sigma=2.0, wa=0):
    import torch
    with F.Plan(torch.from_numpy(np.ascontiguousarray(lam)).cuda(), N, sigma, 6, weight_width=wa) as p:
        return p.weights().cpu().numpy()


@pytest.mark.parametrize("N", [100, 300, 500, 1000])
@pytest.mark.parametrize("periods", [-4096, 65536])
def test_whole_periods_change_nothing(F, N, periods):
    """lambda + k N has the weights of lambda (the coordinates are multiples of 2^-24, so that the sum is
    exact). Bar: the arithmetic's 1e-12 of test_gpu_weights_split."""
    lam = sasgen.random_case(N, 1500, N, spread=min(N, 60))[0]
    lam = np.round(lam * 2.0 ** 24) / 2.0 ** 24
    ref = weights(F, lam, N)
    assert np.max(np.abs(weights(F, lam + periods * N, N) / ref - 1)) < 1e-12
