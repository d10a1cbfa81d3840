"""Exact weights of rasters that the usual ones do not describe: far from the origin, strongly uneven,
window widths and oversamplings whose lag grid is no power of two."""
import os
import subprocess
import sys

import numpy as np
import pytest

import sasgen
from oracle import ftcg_oracle as O

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


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


@pytest.mark.parametrize("N,sigma,wa", [
    (256, 2.5, 4), (200, 3.0, 4), (224, 2.0, 4), (224, 2.0, 6), (224, 2.25, 12), (144, 1.75, 12),
    (100, 2.0, 0), (300, 2.0, 0), (500, 2.0, 0), (200, 1.5, 0), (200, 1.25, 0), (128, 2.0, 4), (64, 4.0, 6),
])
def test_no_less_exact_than_on_the_requested_grid(F, N, sigma, wa):
    """The rms error against pair sums is no larger than that of the FP64 lag route on a grid of side
    2 sigma N, whatever grid the library takes. 10 % and 1e-13 for the two routes' rounding."""
    lam = sasgen.random_case(N + wa, 1500, N, spread=N)[0]
    ref, _ = O.weights_brute(lam, N)
    err = lambda a: np.sqrt(np.mean((a / ref - 1) ** 2))
    assert err(weights(F, lam, N, sigma, wa)) < \
        1.1 * err(O.weights_nufft(lam, N, sigma, wa or 12)[0]) + 1e-13


@pytest.mark.parametrize("N", [512, 1000])
def test_samples_alone_next_to_a_cluster(F, N):
    """300 samples alone in the plane, four million in one spot: the lone samples' S_k are about 1, next to
    4e6 in the cluster. Against pair sums in FP64. Bar: that of test_gpu_weights_split."""
    import torch
    M = 4000000
    rng = np.random.default_rng(N)
    lam = np.concatenate([(rng.random((300, 2)) - 0.5) * N,
                          0.3 + 0.1 * rng.standard_normal((M - 300, 2))])
    k = np.r_[0:300, 300:M:M // 20]
    x, S = torch.from_numpy(lam).cuda(), []
    for c in k:
        d = x - x[c]
        d -= N * torch.round(d / N)
        f = torch.sin(np.pi * (d - torch.round(d))) / (N * torch.sin(np.pi * d / N))
        S.append(torch.where(d == 0, torch.ones_like(d), f).square().prod(1).sum().item())
    tol = 100 * np.exp(-0.97 * np.pi * 0.75 * 12) + 1e-12
    assert np.max(np.abs(weights(F, lam, N)[k] * S - 1)) < tol


def test_little_device_memory(F):
    """N = 1030 with 600 MiB free: too little for the lag grid of side 8192 (672 MB), enough for the one of
    2 sigma N = 4120 (272 MB). In a process of its own, whose memory pool is empty."""
    code = """
import numpy as np, torch
import paper_1706_08575_gb300 as F, sasgen
from oracle import ftcg_oracle as O
lam = sasgen.random_case(3, 300, 1030, spread=60)[0]
with F.Plan(torch.from_numpy(lam).cuda(), 1030, 2.0, 6) as p:
    torch.cuda.synchronize()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (600 << 20), dtype=torch.uint8, device="cuda")
    a = p.weights().cpu().numpy()
assert np.max(np.abs(a / O.weights_brute(lam, 1030)[0] - 1)) < 1e-10
"""
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr


@pytest.mark.parametrize("N", [130, 200, 256])
def test_against_pair_sums_at_lag_side_1024(F, N):
    """Bar of test_gpu_weights_split, which has the other lag grid sides."""
    lam = sasgen.random_case(N, 1500, N, spread=60)[0]
    ref, _ = O.weights_brute(lam, N)
    assert np.max(np.abs(weights(F, lam, N) / ref - 1)) < 100 * np.exp(-0.97 * np.pi * 9.0) + 1e-12


def test_full_accumulators(F):
    """640,000 samples on four lattice points: work items of 1023 samples (from 622 k samples on), each of
    which adds the largest product, 1, to one cell. The lattice points don't see one another, so a weight is
    one over its point's multiplicity."""
    n = np.array([1023, 200000, 318977, 120000])
    pts = np.array([[0.0, 0.0], [3.0, -7.0], [-20.0, 11.0], [31.0, 30.0]])
    which = np.random.default_rng(1).permutation(np.repeat(np.arange(4), n))
    a = weights(F, pts[which], 64)
    assert np.max(np.abs(a * n[which] - 1)) < 100 * np.exp(-0.97 * np.pi * 9.0) + 1e-12
