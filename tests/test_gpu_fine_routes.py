"""Which solve a fine step takes, and each of them where it is taken."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2510_07672_gb300 as G
from test_gpu_mass_sums import random_fields

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
