"""The row-streaming conv at its edges: rows per block of the fused last
layer's projection, fields that start off a 16-byte boundary, and the GELU's
tails and special values."""
import numpy as np
import pytest
import torch

import acpr_inputs as I
import oracle as O
import paper_2510_07672_gb300 as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C", [32, 64])
@pytest.mark.parametrize("batch,act", [(1, 1), (3, 0), (5, 1)])
def test_fused_projection_row_splits(C, batch, act):
    """128 rows a field over the SMs: one row a block, one to three, four to
    five (the projection's two buffers unused, used once, reused).  Tolerance
    of test_cnn_bf16_persistent_shapes; the mass shift sums the same maps."""
    n, L = 128, 4
    w, b = I.cnn_weights(L, C, seed=9, sigma=0.05)
    w32, b32 = w.astype(np.float32), b.astype(np.float32)
    u = np.stack([I.random_field(n, seed=s) for s in range(batch)]).astype(np.float32)
    net = G.CoarseNet(L, C, w32, b32, act=act, precision=G.AC_F32, mass_fix=1)
    got = G.cnn_coarse_step(net, torch.tensor(u, device="cuda")).double().cpu().numpy()
    ref = O.cnn_forward(O.CnnSpec(L, C, w32.astype(np.float64), b32.astype(np.float64), act=act, mass_fix=1, bf16=1),
                        u.astype(np.float64))
    err = np.abs(got - ref)
    scale = max(np.abs(ref - u).max(), 1e-3)
    assert err.max() < 2e-2 * scale + 1e-6
    assert np.median(err) < 1e-3 * scale + 1e-7


@pytest.mark.parametrize("mass", [0, 1])
def test_fields_off_a_vector_boundary(mass):
    """Input and output one float past a 16-byte boundary give the same bits."""
    n, L, C, batch = 128, 3, 32, 2
    w, b = I.cnn_weights(L, C, seed=3, sigma=0.05)
    net = G.CoarseNet(L, C, w.astype(np.float32), b.astype(np.float32), act=1, precision=G.AC_F32, mass_fix=mass)
    u = torch.tensor(np.stack([I.random_field(n, seed=s) for s in range(batch)]), dtype=torch.float32, device="cuda")
    want = G.cnn_coarse_step(net, u)
    src = torch.empty(u.numel() + 1, device="cuda")[1:].view_as(u)
    dst = torch.full((u.numel() + 2,), 7.0, device="cuda")
    src.copy_(u)
    got = G.cnn_coarse_step(net, src, dst[1:-1].view_as(u))
    assert torch.equal(got, want)
    assert float(dst[0]) == 7.0 and float(dst[-1]) == 7.0


@pytest.mark.parametrize("n,L", [(64, 2), (128, 3)])
def test_gelu_tails_and_nan(n, L):
    """A stack that passes bf16(u) through its GELUs (centre taps of channel 0):
    zeros stay zero, large values stay themselves, the far negative tail is
    zero, subnormal-sized values halve, a NaN stays one."""
    C = 32
    w = np.zeros(C * 9 + (L - 2) * C * C * 9 + C * 9)
    w[4] = 1.0
    for l in range(L - 2):
        w[C * 9 + l * C * C * 9 + 4] = 1.0
    w[C * 9 + (L - 2) * C * C * 9 + 4] = 1.0
    b = np.zeros(C * (L - 1) + 1)
    net = G.CoarseNet(L, C, w.astype(np.float32), b.astype(np.float32), act=1, precision=G.AC_F32, residual=0)
    vals = np.array([0.0, -0.0, 8.0, -8.0, 8.5, -8.5, 60.0, -60.0, 1e30, -1e30, 2.0 ** -100, -2.0 ** -100])
    u = np.zeros((1, n, n), dtype=np.float32)
    u[0, 1, 1:2 * len(vals):2] = vals
    u[0, n // 2, n // 2] = np.nan
    got = G.cnn_coarse_step(net, torch.tensor(u, device="cuda")).cpu().numpy()[0]
    assert np.isnan(got[n // 2, n // 2])
    out = got[1, 1:2 * len(vals):2].astype(np.float64)
    half = 2.0 ** -100 * 0.5 ** (L - 1)
    ref = np.array([0, 0, 8, 0, 8.5, 0, 60, 0, float(np.float32(torch.tensor(1e30).to(torch.bfloat16).float())), 0, half, -half])
    assert np.all(np.abs(out - ref) <= 1e-7 + 2.0 ** -8 * np.abs(ref))
    assert np.all(np.abs(out[-2:] / ref[-2:] - 1) < 2.0 ** -7)
