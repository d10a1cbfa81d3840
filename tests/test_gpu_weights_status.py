"""Weight sums that come out <= 0 (narrow windows, whose truncation error next to 20,000 coincident
samples exceeds the 1 that a lone sample adds): reported by the call that first finds one, and again
after ftcg_check has read the plan's status, on both routes of the exact weights."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    import __graft_entry__ as g
    g.build()
    import paper_1706_08575_gb300 as pkg
    return pkg


def status(f):
    try:
        f()
        return 0
    except RuntimeError as e:
        return e.status


@pytest.mark.parametrize("N,sigma,wa", [(64, 2.0, 4), (2050, 2.0, 4)], ids=["pairs", "fp64"])
def test_bad_sums_are_reported_until_checked(F, N, sigma, wa):
    import torch
    spot = np.array([[0.375147, 0.31673817]])
    lam = torch.from_numpy(np.concatenate([np.repeat(spot, 20000, 0), spot + [1.0, 0.0]])).cuda()
    with F.Plan(lam, N, sigma, 4, weight_width=wa) as p:
        assert status(p.weights) == 5
        assert status(p.weights) == 0               # the status is still set
        assert status(p.check) == 5
        assert status(p.check) == 0
        a = torch.empty(20001, dtype=torch.float64, device="cuda")
        assert status(lambda: p.weights(a)) == 5
        assert a[-1].item() == 0.0 and abs(a[0].item() * 20000 - 1) < 1e-2
