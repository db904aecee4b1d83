"""The mass-conserving mean at every scale of the field: flat phases, small,
large, growing and decaying fields, in the kernels that form the sums of the
right-hand side in integers (fine_stencil.cu, fine_tiles.cu)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import acpr_inputs as I
import paper_2510_07672_gb300 as G

pytestmark = pytest.mark.gpu

F32, F64 = G.AC_F32, G.AC_F64


def params(n, prec, lam, dt=1e-4, S=2.0):
    """lam = dt eps^2 4 / h^2; mass-conserving."""
    return G.FineParams(n, float(np.sqrt(lam / (4 * dt))) / n, S, dt, variant=G.AC_MASS_CONSERVING, precision=prec)


def propagate(fp, steps, u):
    return (G.ac_fine3d_propagate if u.dim() == 4 else G.ac_fine_propagate_slices)(fp, steps, u)


def mean(u):
    return u.double().mean(dim=tuple(range(1, u.dim())))


def random_fields(shape, dtype, seed=1):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.rand(shape, generator=g, device="cuda", dtype=dtype) * 1.8 - 0.9


def field_ref(u, fp, steps):
    """The step with a float64 Fourier solve, 2D or 3D."""
    n, dims = fp.n, u.dim() - 1
    axes = tuple(range(1, dims + 1))
    s2 = torch.sin(torch.pi * torch.arange(n, device="cuda", dtype=torch.float64) / n) ** 2
    a = 1 + fp.S * fp.dt
    sym = a
    for d in range(dims):
        m = s2[: n // 2 + 1] if d == dims - 1 else s2
        sym = sym + fp.dt * fp.eps ** 2 * 4 * n * n * m.reshape([-1 if d == b else 1 for b in range(dims)])
    v = u.double()
    for _ in range(steps):
        f = v - v ** 3
        if fp.variant:
            f = f - f.mean(dim=axes, keepdim=True)
        v = torch.fft.irfftn(torch.fft.rfftn(a * v + fp.dt * f, dim=axes) / sym, s=(n,) * dims, dim=axes)
    return v


GRIDS32 = [(32, 2), (64, 2), (128, 2), (256, 2), (512, 2), (1024, 2), (32, 3), (64, 3), (128, 3)]
VALUES = [0.1, 0.9713, -0.9421, 0.9067, 0.9951, 1.1e-3, 1.7e-8, 3e-20]


@pytest.mark.parametrize("steps", [1, 2, 5])
@pytest.mark.parametrize("n,dims", GRIDS32)
def test_flat_fields_stay(n, dims, steps):
    """A constant field is a fixed point: f - mean f = 0.  One ulp: the two
    roundings of the last step (half an ulp each) around the exact mean."""
    fp = params(n, F32, 1.25e-3)
    c = torch.tensor(VALUES, dtype=torch.float32, device="cuda")
    u = c.reshape((-1,) + (1,) * dims).expand((-1,) + (n,) * dims).contiguous()
    err = (propagate(fp, steps, u).double() - u.double()).abs().amax(dim=tuple(range(1, dims + 1))).cpu().numpy()
    assert np.all(err <= np.spacing(np.abs(np.float32(VALUES)))), err


@pytest.mark.parametrize("n,lam", [(32, 8e-4), (64, 8e-4), (128, 3e-3), (256, 8e-3)])
def test_flat_fields_stay_f64(n, lam):
    """float64: four ulp (the rounded sums of u and of r, three roundings each,
    and the last step's two)."""
    fp = params(n, F64, lam)
    vals = np.array([0.1, -0.9421, 1.2345e-8, 3e-200])
    u = torch.tensor(vals, device="cuda").reshape(-1, 1, 1).expand(-1, n, n).contiguous()
    err = (propagate(fp, 3, u) - u).abs().amax(dim=(1, 2)).cpu().numpy()
    assert np.all(err <= 4 * np.spacing(np.abs(vals))), err


@pytest.mark.parametrize("n,dims", GRIDS32)
def test_small_fields_keep_their_mean(n, dims):
    """Noise of size 1e-6 about 5e-7: the mean moves by less than the rounding
    of one cell (2^-25 of the largest), the bound of a rounding bias."""
    fp = params(n, F32, 1.25e-3)
    u = random_fields((2,) + (n,) * dims, torch.float32) * 1e-6 + 5e-7
    out = propagate(fp, 5, u)
    assert (mean(out) - mean(u)).abs().max().item() <= 2.0 ** -25 * u.abs().max().item()


@pytest.mark.parametrize("n,dims,prec", [g + (F32,) for g in GRIDS32] + [(32, 2, F64), (64, 2, F64), (256, 2, F64)])
def test_large_fields(n, dims, prec):
    """Fields of size 2^21 at a step that resolves them: against 64 bits, the
    round-off of the comparison at size one."""
    size = 2.0 ** 21
    fp = params(n, prec, 1e-3, dt=1e-3 / size ** 2)
    u = random_fields((2,) + (n,) * dims, torch.float64 if prec == F64 else torch.float32) * size
    out = propagate(fp, 3, u)
    tol = 1e-14 if prec == F64 else 1.2e-7 * 4
    assert (out.double() - field_ref(u, fp, 3)).abs().max().item() < tol * size


@pytest.mark.parametrize("n,prec", [(32, F32), (128, F32)])
def test_growing_noise(n, prec):
    """Noise of 1e-6 grows by e^16 within one call.  Relative to the float64
    Fourier solve: each of 1600 steps rounds twice, all grow alike."""
    dt, steps = 1e-2, 1600
    fp = params(n, prec, 1e-3, dt=dt)
    u = random_fields((2, n, n), torch.float32) * 1e-6
    out = propagate(fp, steps, u)
    ref = field_ref(u, fp, steps)
    assert ref.abs().max().item() > 0.1
    assert (out.double() - ref).abs().max().item() < steps * 2 * 2.0 ** -23


@pytest.mark.parametrize("n,dims", GRIDS32)
def test_decaying_field_keeps_a_small_mean(n, dims):
    """A checkerboard of 0.75 about 2^-23 decays within one call to the ripple
    that rounding holds up (0.009 of it below half an ulp); its mean is the
    entry mean to one ulp, as above."""
    lam = 4.5e-3 if dims == 2 else 3e-3
    fp = params(n, F32, lam, dt=1e-6)
    i = torch.arange(n, device="cuda")
    par = i.reshape(-1, 1) + i
    if dims == 3:
        par = par.reshape(n, n, 1) + i
    c = 2.0 ** -23
    u = (0.75 * (1 - 2 * (par % 2)).float() + c)[None].contiguous()
    out = propagate(fp, 5000, u)
    ulp = float(np.spacing(np.float32(c)))
    assert (out - c).abs().max().item() <= 60 * ulp
    assert (mean(out) - c).abs().item() <= ulp


@pytest.mark.parametrize("n", [32, 64])
def test_adjoint_of_a_growing_mode_f64(n):
    """lambda grows by e^19 through states of zero: the Fourier solve's, to the
    rounding of 2000 steps."""
    steps = 2000
    fp = params(n, F64, 8e-4, dt=1e-2)
    states = torch.zeros((steps, 1, n, n), dtype=torch.float64, device="cuda")
    lam = torch.tensor(I.random_field(n, seed=4)[None], device="cuda")
    got = G.ac_fine_adjoint(fp, steps, states, lam)
    G.ac_fine_set_variant(n, F64, 1)
    try:
        ref = G.ac_fine_adjoint(fp, steps, states, lam)
    finally:
        G.ac_fine_set_variant(n, F64, 0)
    assert ref.abs().max().item() > 2.0 ** 21
    assert (got - ref).abs().max().item() < steps * 2.0 ** -50 * ref.abs().max().item()


@pytest.mark.parametrize("n,prec", [(64, F32), (128, F32), (256, F32), (64, F64)])
def test_batch_size_does_not_change_the_bits(n, prec):
    """Small growing fields, so that the unit of the sums changes on the way:
    every split of the field takes the same units."""
    fp = params(n, prec, 8e-4, dt=5e-2)
    count = 100 if n <= 128 else 40
    u = random_fields((count, n, n), torch.float64 if prec == F64 else torch.float32) * 3e-5 + 1e-5
    full = G.ac_fine_propagate_slices(fp, 70, u)
    for m in (1, 9, 20):
        assert torch.equal(G.ac_fine_propagate_slices(fp, 70, u[:m].clone()), full[:m])
