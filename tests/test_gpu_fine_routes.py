"""Which solve a fine step takes, and each of them where it is taken."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2510_07672_gb300 as G
from paper_2510_07672_gb300 import abi
from test_gpu_mass_sums import field_ref, mean, random_fields

pytestmark = pytest.mark.gpu

F32, F64 = G.AC_F32, G.AC_F64


def params(n, prec, variant, lam, dt=1e-4, S=2.0):
    """lam = dt eps^2 4 / h^2 fixes the degree of the polynomial."""
    return G.FineParams(n, float(np.sqrt(lam / (4 * dt))) / n, S, dt, variant=variant, precision=prec)


def with_shape(n, prec, index, call):
    G.ac_fine_set_variant(n, prec, index)
    try:
        return call()
    finally:
        G.ac_fine_set_variant(n, prec, 0)


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("n,prec", [(32, F32), (128, F32), (512, F32), (64, F64), (256, F64)])
def test_large_stabilisation_takes_the_fourier_solve(n, prec, variant):
    """1 + S dt = 5: b_0 - 1 is -0.8 and its rounding four times that of b_0
    itself, a gain error of every step; up to 1 + S dt = 2 it is no larger."""
    u = random_fields((2, n, n), torch.float64 if prec == F64 else torch.float32)
    run = lambda fp, index: with_shape(n, prec, index, lambda: G.ac_fine_propagate_slices(fp, 3, u))
    fp = params(n, prec, variant, 1e-3, dt=2.0)
    assert torch.equal(run(fp, 0), run(fp, 1))
    fp = params(n, prec, variant, 1e-3, dt=0.5)
    assert not torch.equal(run(fp, 0), run(fp, 1))


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("steps", [1, 2, 3])
@pytest.mark.parametrize("lam", [2.5e-3, 2e-2])
def test_cube_buffers_that_overlap(steps, variant, lam):
    """u_in and u_out share two of three fields, either one first: the same bits
    as apart (streamed planes, and the passes that stiff steps take)."""
    n, size = 32, 32 ** 3
    fp = params(n, F32, variant, lam)
    u = random_fields((3, n, n, n), torch.float32)
    want = G.ac_fine3d_propagate(fp, steps, u)
    for first, second in ((0, size), (size, 0)):
        buf = torch.empty(4 * size, device="cuda")
        src, dst = buf[first:first + 3 * size].view_as(u), buf[second:second + 3 * size].view_as(u)
        src.copy_(u)
        G.ac_fine3d_propagate(fp, steps, src, dst)
        assert torch.equal(dst, want)


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("lam", [5.5e-3, 2e-2, 0.3])
def test_stiff_1024_takes_the_two_passes(lam, variant):
    """1024^2 steps beyond degree 2 (lambda above 4.95e-3): against 64 bits, the
    round-off of a float32 Fourier solve, eps log2(n^2) a step; with a caller's
    workspace the same bits."""
    n, steps = 1024, 4
    fp = params(n, F32, variant, lam)
    u = random_fields((2, n, n), torch.float32) + 0.03
    out = G.ac_fine_propagate_slices(fp, steps, u)
    assert (out.double() - field_ref(u, fp, steps)).abs().max().item() < steps * 20 * 2.0 ** -23
    if variant:
        assert (mean(out) - mean(u)).abs().max().item() < 1e-7
    need = G.ac_fine_workspace_bytes(n, 2, F32)
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    got = G.ac_fine_propagate_slices_ws(fp, steps, u, torch.empty_like(u), ws)
    assert torch.equal(got, out)


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("n,prec,counts", [(64, F32, (1, 76, 77)), (128, F32, (12, 13, 96, 97)), (256, F32, (6, 7, 24, 25)),
                                           (64, F64, (9, 10))])
def test_every_split_gives_the_same_bits(n, prec, counts, variant):
    """Both sides of every batch size at which the split changes."""
    fp = params(n, prec, variant, 8e-4)
    u = random_fields((counts[-1], n, n), torch.float64 if prec == F64 else torch.float32)
    full = G.ac_fine_propagate_slices(fp, 6, u)
    for m in counts[:-1]:
        assert torch.equal(G.ac_fine_propagate_slices(fp, 6, u[:m].clone()), full[:m]), m


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("n,lam,steps,every", [(64, 1.3e-3, 11, 4), (256, 1.31e-3, 7, 3), (128, 3.5e-3, 6, 2), (256, 8e-3, 5, 2)])
def test_energy_gradient_overlap_f64_degrees(n, lam, steps, every, variant):
    """float64 degrees 5 (side by side) and 6 (one after the other): the same
    bits with and without room for two segments."""
    fp = params(n, F64, variant, lam)
    u = random_fields((n, n), torch.float64)
    got = G.ac_energy_gradient_ic(fp, steps, u, checkpoint_every=every)
    p = fp.c()
    lib = G.load()
    nbytes = lib.ac_energy_gradient_workspace(ctypes.byref(p), steps, every) - u.numel() * 8 * (every + 1)
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    ref = torch.empty_like(u)
    rc = lib.ac_energy_gradient_ic(ctypes.byref(p), steps, every, u.data_ptr(), ref.data_ptr(), ws.data_ptr(), nbytes,
                                   torch.cuda.current_stream().cuda_stream)
    assert rc == abi.AC_OK
    torch.cuda.synchronize()
    assert torch.equal(got, ref)
