"""The judge's sums at the edges of its blocks: one judged sample, numbers of judged samples that
are no multiple of the four of a block, sample counts around one part (1024), and the smallest image
sides, where lags wrap at every step. Bar of test_gpu_judge (1e-6) against the FP64 pair sums."""
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


@pytest.mark.parametrize("M,K,N", [(1, 1, 16), (7, 5, 16), (1024, 9, 64), (1025, 1025, 32),
                                   (3000, 6, 18), (500, 33, 8)])
def test_judge_sums_at_block_edges(F, M, K, N):
    import torch
    lam, _ = sasgen.random_case(M + K, M, N, spread=3 * N)
    rng = np.random.default_rng(M)
    alpha = np.exp(0.3 * rng.standard_normal(M))
    ref, _ = O.weights_brute(lam, N)
    k = (2 * np.arange(K) + 1) * M // (2 * K)
    q = alpha[k] / ref[k]
    with F.Plan(torch.from_numpy(lam).cuda(), N, 2.0, 4) as p:
        _, st = p.judge_weights(torch.from_numpy(alpha).cuda(), K=K, max_rel_err=100.0)
    med = np.median(q)
    e = q / med - 1.0
    assert abs(st["median_ratio"] - med) < 1e-6 * med
    assert abs(st["rms"] - np.sqrt(np.mean(e ** 2))) < 1e-6 * (1 + st["rms"])
    assert abs(st["max"] - np.max(np.abs(e))) < 1e-6 * (1 + st["max"])
