"""The fused training kernel at the edges of its 64-row tiles: one row, one row short of a tile, a
full tile, one more, and more tiles than resident CTAs, through an index with repeated rows and with
features at a 4-byte offset. Bars as in test_gpu_mlp (4 E + 1e-5 of the FP64 oracle, E the error
that the device's six bfloat16 roundings cause on their own)."""
import numpy as np
import pytest

from oracle import mlp_oracle as L
from test_gpu_mlp import bf16, bf16_model, dev, nrel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    import __graft_entry__ as g
    g.build()
    import paper_1706_08575_gb300 as pkg
    return pkg


@pytest.mark.parametrize("B,indexed,offset", [(1, False, 0), (63, True, 0), (64, False, 2),
                                              (65, True, 2), (64 * 304 + 17, True, 0)])
def test_grads_at_tile_edges(F, B, indexed, offset):
    import torch
    rng = np.random.default_rng(B)
    P = L.init_params(rng)
    P["w4"] = rng.standard_normal(L.HID) * 0.2
    P["b1"] = rng.standard_normal(L.HID) * 0.1
    flat = L.pack(P).astype(np.float32)
    rows = 500 if indexed else B
    X = bf16(rng.standard_normal((rows, L.D_IN)) * 0.7)
    t = rng.standard_normal(rows) * 0.5
    buf = torch.zeros(rows * 48 + offset, dtype=torch.bfloat16, device="cuda")
    Xt = buf[offset:].view(rows, 48)
    Xt[:, :L.D_IN] = torch.from_numpy(X.astype(np.float32)).to(torch.bfloat16).cuda()
    idx = rng.integers(0, rows, B) if indexed else np.arange(B)
    it = torch.from_numpy(idx.astype(np.int32)).cuda() if indexed else None
    mlp = F.Mlp(flat)
    g, loss = mlp.grads(Xt, dev(t), it)
    g2, loss2 = mlp.grads(Xt, dev(t), it)
    mlp.close()
    assert np.array_equal(g, g2) and loss == loss2
    Pr = L.unpack(flat)
    for k in ("W1", "W2", "W3", "w4"):
        Pr[k] = bf16(Pr[k])
    y_ref, cache = L.forward(Pr, X[idx])
    g_ref, l_ref = L.backward(Pr, cache, y_ref, t[idx]), L.loss(y_ref, t[idx])
    _, g_m, l_m = bf16_model(Pr, X[idx], t[idx])
    assert abs(loss - l_ref) / l_ref <= 4 * abs(l_m - l_ref) / l_ref + 1e-5
    G = L.unpack(g)
    for k, _ in L.ORDER:
        assert nrel(G[k], g_ref[k]) <= 4 * nrel(g_m[k], g_ref[k]) + 1e-5, k
