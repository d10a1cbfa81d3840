"""The adjoint through cuFFT (grid sides that are no power of two, so never the shared-memory transforms):
captured in a CUDA graph, from host buffers, one call and a pipeline of calls. Bars of test_gpu_parity."""
import numpy as np
import pytest

import sasgen
from oracle import ftcg_oracle as O

pytestmark = pytest.mark.gpu
SIDES = [36, 72, 100]


@pytest.fixture(scope="module")
def F():
    import __graft_entry__ as g
    g.build()
    import paper_1706_08575_gb300 as pkg
    return pkg


def dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def plan(F, lam, N):
    p = F.Plan(dev(lam), N, 2.0, 8)
    assert p.G & (p.G - 1) != 0
    return p


@pytest.mark.parametrize("N", SIDES)
def test_captured_in_cuda_graph(F, N):
    import torch
    lam, v = sasgen.random_case(61, 3000, N, spread=N)
    v2 = (np.random.default_rng(62).standard_normal(3000) + 1j).astype(np.complex64)
    with plan(F, lam, N) as p:
        vals = dev(v.astype(np.complex64))
        img = torch.zeros((N, N), dtype=torch.complex64, device="cuda")
        p.adjoint(vals, out=img)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            p.adjoint(vals, out=img)
        vals.copy_(dev(v2))
        img.zero_()
        g.replay()
        torch.cuda.synchronize()
        got = img.cpu().numpy()
    assert O.rel_l2(got, O.adjoint(lam, v2.astype(np.complex128), N, 2.0, 8)) < 1e-5


@pytest.mark.parametrize("N", SIDES)
@pytest.mark.parametrize("pinned", [True, False], ids=["pinned", "pageable"])
def test_host_buffers(F, N, pinned):
    import torch
    lam, _ = sasgen.random_case(51, 2000, N, spread=N)
    rng = np.random.default_rng(N)
    vs = [(rng.standard_normal(2000) + 1j * rng.standard_normal(2000)).astype(np.complex64)
          for _ in range(4)]
    put = (lambda t: t.pin_memory()) if pinned else (lambda t: t)
    with plan(F, lam, N) as p:
        refs = [p.adjoint(dev(v)).cpu().numpy() for v in vs]
        hv = [put(torch.from_numpy(v)) for v in vs]
        one = put(torch.full((N, N), 7.0 + 0j, dtype=torch.complex64))
        p.adjoint_host(hv[0], one)
        imgs = [put(torch.full((N, N), 7.0 + 0j, dtype=torch.complex64)) for _ in vs]
        s = torch.cuda.Stream()
        for h, i in zip(hv, imgs):
            p.adjoint_host_async(h, i, stream=s)
        s.synchronize()
    assert O.rel_l2(one.numpy(), refs[0]) < 1e-6
    for i, r in zip(imgs, refs):
        assert O.rel_l2(i.numpy(), r) < 1e-6
