"""The exact weights' route without the FP64 pipe where it can go wrong: every lag grid side (256 to
8192), N that is no power of two, narrow and odd weight windows, samples on ties and far outside one
period; and the routes next to it that stay on
FP64 (wide windows, large sigma). Against weights summed pair by pair in FP64. Tolerance: the
lag route's error is its window's truncation, of the order exp(-beta) amplified by the window
division by less than 100 on these rasters; the arithmetic's 1e-12 is added."""
import math

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


def raster(kind, N, seed):
    rng = np.random.default_rng(seed)
    if kind == "uniform":
        return sasgen.random_case(seed, 1500, N, spread=min(N, 60))[0]
    if kind == "ties":                       # multiples of 1/8 cycle, several periods away
        lam = rng.integers(-8 * 20, 8 * 20, (900, 2)) / 8.0
        return lam + N * rng.integers(-3, 4, (900, 2))
    # beyond the 16-bit range of the position words
    return sasgen.random_case(seed, 600, N, spread=20)[0] + N * 70000.0


@pytest.mark.parametrize("N,sigma,wa,kind", [
    (32, 2.0, 0, "uniform"), (64, 2.0, 0, "ties"), (100, 2.0, 0, "uniform"),
    (128, 1.25, 0, "uniform"), (500, 2.0, 11, "uniform"),
    (640, 1.5, 7, "ties"), (1024, 2.0, 4, "uniform"), (1100, 2.0, 0, "uniform"),
    (64, 2.0, 0, "far"), (64, 2.0, 14, "uniform"), (64, 3.0, 0, "uniform"),
])
def test_weights_against_pair_sums(F, N, sigma, wa, kind):
    import torch
    lam = raster(kind, N, N + wa)
    w = wa or 12
    tol = 100 * math.exp(-0.97 * math.pi * (1 - 0.5 / sigma) * w) + 1e-12
    if kind == "far":                        # the FP64 coordinate itself: 70000 N rounded to 2^-31
        tol += 1e-7
    with F.Plan(torch.from_numpy(lam).cuda(), N, sigma, 6, weight_width=wa) as p:
        got = p.weights().cpu().numpy()
        again = p.weights().cpu().numpy()
    ref, _ = O.weights_brute(lam, N)
    assert np.max(np.abs(got - ref) / ref) < tol
    assert np.max(np.abs(got - again) / ref) < 1e-12
