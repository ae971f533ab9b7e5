"""The network's dense products at the edges of their tiles and chunks (odd and
even chunk counts, a remainder of K, rows that 128-bit loads cannot take,
tiles partly outside the output) and the fused backward sums, against the FP64
oracle on the same bfloat16-rounded operands, with the bars of
test_gpu_mlp.py."""
import numpy as np
import pytest
import torch

import oracle.learned as L

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,F,H", [(512, 4096, 256), (130, 1030, 65), (1000, 2049, 100),
                                   (129, 512, 63), (31, 64, 7), (300, 65, 513), (5, 1, 1)])
def test_products_and_gradients(n, F, H):
    from paper_1905_13257_gb300 import Mlp
    from paper_1905_13257_gb300 import _binding as B
    rng = np.random.default_rng(n + F + H)
    X = rng.standard_normal((n, F)).astype(np.float32)
    y = (rng.random(n) < 0.2).astype(np.float64)
    p = L.init_params(F, H, seed=4)
    p["b1"] = rng.standard_normal(H) * 0.2
    p["b2"] = 0.05
    p = {k: np.asarray(v, dtype=np.float32).astype(np.float64) for k, v in p.items()}
    net = Mlp(p)
    Xd = torch.from_numpy(X).cuda()
    s = net.forward(Xd).cpu().numpy()
    so, (Zo, Go) = L.forward(X.astype(np.float64), p, product_round=L.bf16_operands)
    assert np.max(np.abs(s - so)) <= 1e-5 * max(1.0, np.abs(so).max())
    assert np.max(np.abs(net.G.cpu().numpy() - Go)) <= 1e-5 * max(1.0, np.abs(Go).max())
    go = L.backward(X.astype(np.float64), y, p, 3.0, product_round=L.bf16_operands)
    # through the C call, which leaves dZ with the caller: the W1 gradient is
    # compared with the exact product of the dZ the kernels formed (a dZ that
    # lies on a rounding boundary of bfloat16 may round either way)
    f32 = dict(dtype=torch.float32, device="cuda")
    g = {"W1": torch.empty(F, H, **f32), "b1": torch.empty(H, **f32), "w2": torch.empty(H, **f32),
         "b2": torch.empty(1, **f32)}
    ds, dZ, yd = torch.empty(n, **f32), torch.empty(n, H, **f32), torch.tensor(y, **f32)
    ptr = lambda t: B.C.c_void_p(t.data_ptr())   # noqa: E731
    assert net.lib.id_mlp_backward(ptr(Xd), n, F, H, ptr(net.Z), ptr(net.G), ptr(net.w2),
                                   ptr(net.s), ptr(yd), 3.0, ptr(g["W1"]), ptr(g["b1"]),
                                   ptr(g["w2"]), ptr(g["b2"]), ptr(ds), ptr(dZ), net._sh) == 0
    go["W1"] = L.bf16_operands(X.astype(np.float64)).T @ \
        L.bf16_operands(dZ.cpu().numpy().astype(np.float64))
    for key in ("W1", "b1", "w2", "b2"):
        a = g[key].cpu().numpy().reshape(-1)
        b = np.atleast_1d(np.asarray(go[key], dtype=np.float64)).reshape(-1)
        assert np.max(np.abs(a - b)) <= 1e-4 * np.abs(b).max(), key
    net.check()
