"""The judge's sums at samples that nearly coincide: both axes' factors of such a lag are tiny, their
products far below the FP32 range, while the Fejer kernel is 1. The prediction of the two samples is
wrong by a factor of three, so that the verdict changes if a sum of theirs is lost. Bar of
test_gpu_judge (1e-6) against the FP64 pair sums."""
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


@pytest.mark.parametrize("N", [8, 64, 1024, 4096])
@pytest.mark.parametrize("lag", [(1e-22, 1e-22), (2e-14, 1e-30), (4e-16, 2.7e-32), (1e-13, 1e-13),
                                 (2e-12, 2e-12), (1e-3, 1e-40), (0.0, 1e-25), (1e-7, 3e-6)])
def test_near_coincident_samples(F, lag, N):
    import torch
    lam = np.concatenate([sasgen.random_case(N, 200, N, spread=N)[0], [[0.0, 0.0], lag]])
    M = len(lam)
    ref, _ = O.weights_brute(lam, N)
    alpha = ref.copy()
    alpha[-2:] *= 3.0
    with F.Plan(torch.from_numpy(lam).cuda(), N, 2.0, 4) as p:
        _, st = p.judge_weights(torch.from_numpy(alpha).cuda(), K=M, max_rel_err=100.0)
    e = alpha / ref - 1.0                    # the median ratio is 1
    assert abs(st["median_ratio"] - 1.0) < 1e-6
    assert abs(st["rms"] - np.sqrt(np.mean(e ** 2))) < 1e-6 * (1 + st["rms"])
    assert abs(st["max"] - 2.0) < 1e-6 * 3
