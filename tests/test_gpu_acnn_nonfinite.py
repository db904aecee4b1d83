"""The ACNN's mass shift when a field holds an infinity: the float32 network
gives what the float64 one gives."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import acpr_inputs as I
import paper_2510_07672_gb300 as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C", [4, 16])
@pytest.mark.parametrize("bad", [float("inf"), -float("inf"), float("nan")])
@pytest.mark.parametrize("limiter", [0, 1])
def test_mass_shift_of_an_infinite_field(C, bad, limiter):
    """tanh keeps the layers finite, so the shift is the infinity: every cell
    becomes one, or the limiter's bound.  The other field is not touched."""
    n = 32
    w, b = I.acnn_weights(C, 1, seed=3)
    u = np.stack([I.random_field(n, seed=s) for s in range(2)])
    u[0, 5, 7] = bad
    res = []
    for prec, dt in ((G.AC_F32, torch.float32), (G.AC_F64, torch.float64)):
        net = G.Acnn(C, 1, w, b, mass_fix=1, limiter=limiter, lo=-1.0, hi=1.0, precision=prec)
        ut = torch.tensor(u, dtype=dt, device="cuda")
        res.append([net(ut).double(), net.forward_train(ut, net.new_workspace(n, 2)).double()])
    for a, ref in zip(*res):
        assert torch.equal(a[0].isnan(), ref[0].isnan())
        assert torch.equal(a[0].nan_to_num(9.0, 1e9, -1e9), ref[0].nan_to_num(9.0, 1e9, -1e9))
        assert torch.allclose(a[1], ref[1], rtol=0, atol=1e-5)
