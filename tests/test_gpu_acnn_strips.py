"""The strip kernels of the float32 C = 4 ACNN (forward, input gradients,
weight gradients) against the float64 network at the smallest and odd sizes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import acpr_inputs as I
import paper_2510_07672_gb300 as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,batch,blocks,mass", [(32, 1, 0, 0), (32, 3, 2, 1), (64, 1, 1, 1), (64, 5, 3, 0), (128, 2, 4, 1),
                                                 (512, 1, 2, 1)])
def test_strips_match_float64(n, batch, blocks, mass):
    """Tolerances: float32 sums of 9 C terms through 2 blocks + 2 layers, 1e-5
    of the largest value; gradients sum n^2 products, 1e-4 of the largest."""
    w, b = I.acnn_weights(4, blocks, seed=3)
    u = np.stack([I.random_field(n, seed=s, zero_mean=True) for s in range(batch)])
    gout = np.random.default_rng(5).standard_normal((batch, n, n))
    res = []
    for prec, dt in ((G.AC_F32, torch.float32), (G.AC_F64, torch.float64)):
        net = G.Acnn(4, blocks, w, b, mass_fix=mass, limiter=1, lo=-10.0, hi=10.0, precision=prec)
        ut, gt = torch.tensor(u, dtype=dt, device="cuda"), torch.tensor(gout, dtype=dt, device="cuda")
        ws = net.new_workspace(n, batch)
        out = net.forward_train(ut, ws)
        gw, gb = net.backward(ut, gt, ws)
        res.append([x.double() for x in (out, gw, gb)])
        gw2, gb2 = net.backward(ut, gt, ws)
        assert torch.equal(gw, gw2) and torch.equal(gb, gb2)
    for k, (a, ref) in enumerate(zip(*res)):
        assert (a - ref).abs().max().item() < (1e-4 if k else 1e-5) * max(ref.abs().max().item(), 1e-3), k
