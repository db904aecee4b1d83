"""The polynomial solve of the fine step (fine_stencil.cu, the first launch
shape) against the Fourier solve (the other shapes) over the forms it accepts:
every size, degree, model, batch split, trajectories and adjoints."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import acpr_inputs as I
import paper_2510_07672_gb300 as G

pytestmark = pytest.mark.gpu

F32, F64 = G.AC_F32, G.AC_F64


def fields(n, count, prec, amp=0.9, shift=0.0):
    u = np.stack([I.random_field(n, seed=300 + s, amp=amp) for s in range(count)]) + shift
    return torch.tensor(u, dtype=torch.float64 if prec == F64 else torch.float32, device="cuda")


def with_shape(n, prec, index, call):
    G.ac_fine_set_variant(n, prec, index)
    try:
        return call()
    finally:
        G.ac_fine_set_variant(n, prec, 0)


def params(n, prec, variant, lam, dt=1e-4):
    """lam = dt eps^2 4 / h^2 fixes the degree of the polynomial."""
    return G.FineParams(n, float(np.sqrt(lam / (4 * dt))) / n, 2.0, dt, variant=variant, precision=prec)


# lam: float32 degrees 2, 3, 4 below 4.9e-3, 2.2e-2, 5.5e-2 (512: up to 3); float64 degrees 4, 5, 6 below 1.1e-3, 3.8e-3, 1e-2
CASES = [(n, F32, lam) for n in (32, 64, 128, 256, 512) for lam in (1.25e-3, 1e-2, 3e-2)]
CASES += [(n, F64, lam) for n in (32, 64, 128, 256) for lam in (8e-4, 3e-3, 8e-3)]


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("n,prec,lam", CASES)
def test_matches_the_fourier_solve(n, prec, lam, variant):
    """5 steps.  Tolerance: the round-off of the float32 Fourier solve, about
    eps log2(n^2) |u| = 2e-6 a step at most; float64 the same with its eps."""
    fp = params(n, prec, variant, lam)
    u = fields(n, 3, prec, shift=0.05)
    a = with_shape(n, prec, 0, lambda: G.ac_fine_propagate_slices(fp, 5, u))
    b = with_shape(n, prec, 1, lambda: G.ac_fine_propagate_slices(fp, 5, u))
    assert (a - b).abs().max().item() < (1e-14 if prec == F64 else 1e-5)
    if variant:
        drift = (a.double().mean(dim=(1, 2)) - u.double().mean(dim=(1, 2))).abs().max().item()
        assert drift < (1e-15 if prec == F64 else 1e-8)


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("n,prec", [(32, F32), (64, F32), (128, F32), (256, F32), (512, F32), (64, F64), (128, F64)])
def test_batch_size_does_not_change_the_bits(n, prec, variant):
    """The split over warps and CTAs follows the batch size; a field's result
    does not (Parareal's F and the sequential solve are one function)."""
    count = 80 if n <= 256 else 24
    fp = params(n, prec, variant, 8e-4)
    u = fields(n, count, prec)
    full = G.ac_fine_propagate_slices(fp, 6, u)
    for f in (0, 1, count - 1):
        assert torch.equal(G.ac_fine_propagate_slices(fp, 6, u[f:f + 1].clone())[0], full[f])
    work = torch.tensor([[f, count - 1 - f, 6, 0] for f in range(count)], dtype=torch.int32, device="cuda")
    out = torch.empty_like(u)
    G.ac_fine_propagate_work(fp, work, u, out)
    assert torch.equal(out.flip(0), full)
    traj = G.ac_fine_trajectory(fp, 6, u[:3].clone())
    assert torch.equal(traj[0], u[:3]) and torch.equal(traj[6], full[:3])
    assert torch.equal(traj[2], G.ac_fine_propagate_slices(fp, 2, u[:3].clone()))


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("n,prec", [(32, F32), (64, F32), (128, F32), (256, F32), (512, F32), (32, F64), (64, F64), (256, F64)])
def test_adjoint_matches_the_fourier_solve(n, prec, variant):
    """lambda of any scale (here 1e-6): relative to its largest value, the
    tolerance of the forward comparison."""
    fp = params(n, prec, variant, 1.25e-3)
    u = fields(n, 2, prec)
    states = G.ac_fine_trajectory(fp, 4, u)[:4].contiguous()
    lam = fields(n, 2, prec, amp=0.5, shift=0.2) * 1e-6
    a = with_shape(n, prec, 0, lambda: G.ac_fine_adjoint(fp, 4, states, lam))
    b = with_shape(n, prec, 1, lambda: G.ac_fine_adjoint(fp, 4, states, lam))
    assert (a - b).abs().max().item() < (1e-14 if prec == F64 else 1e-5) * lam.abs().max().item()


def test_stiff_steps_take_the_fourier_solve():
    n = 128
    for prec in (F32, F64):
        fp = params(n, prec, 0, 0.25, dt=1e-2)
        u = fields(n, 2, prec)
        a = with_shape(n, prec, 0, lambda: G.ac_fine_propagate_slices(fp, 3, u))
        assert torch.equal(a, with_shape(n, prec, 1, lambda: G.ac_fine_propagate_slices(fp, 3, u)))


def test_no_diffusion_and_not_a_number():
    n = 64
    for prec in (F32, F64):
        fp = G.FineParams(n, 0.0, 2.0, 1e-4, precision=prec)  # eps = 0: A is a multiple of the identity
        u = fields(n, 2, prec)
        ref = u.double()
        for _ in range(3):
            ref = (1.0002 * ref + 1e-4 * (ref - ref ** 3)) / 1.0002
        assert (G.ac_fine_propagate_slices(fp, 3, u).double() - ref).abs().max().item() < (1e-15 if prec == F64 else 3e-7)
        for bad in (float("nan"), float("inf")):
            v = u.clone()
            v[1, 5, 7] = bad
            for variant in (0, 1):
                out = G.ac_fine_propagate_slices(params(n, prec, variant, 1e-3), 2, v)
                assert torch.isfinite(out[0]).all() and not torch.isfinite(out[1]).all()
                if variant:  # the mean is not a number
                    assert torch.isnan(out[1]).all()


def field_ref(u, fp, steps):
    """The step with a float64 Fourier solve, 2D or 3D."""
    n, dims = fp.n, u.dim() - 1
    axes = tuple(range(1, dims + 1))
    s2 = torch.sin(torch.pi * torch.arange(n, device="cuda", dtype=torch.float64) / n) ** 2
    sym = 1 + fp.S * fp.dt
    for a in range(dims):
        m = s2[: n // 2 + 1] if a == dims - 1 else s2
        sym = sym + fp.dt * fp.eps ** 2 * 4 * n * n * m.reshape([-1 if a == b else 1 for b in range(dims)])
    v = u.double()
    for _ in range(steps):
        f = v - v ** 3
        if fp.variant:
            f = f - f.mean(dim=axes, keepdim=True)
        v = torch.fft.irfftn(torch.fft.rfftn((1 + fp.S * fp.dt) * v + fp.dt * f, dim=axes) / sym, s=(n,) * dims, dim=axes)
    return v


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("steps", [1, 3, 4, 5, 9])
def test_tiles_1024(steps, variant):
    """One to three launches of up to four steps, every tile edge: against
    float64.  Tolerance: two roundings of values below 1 a step."""
    n = 1024
    fp = G.FineParams(n, 0.004, 2.0, 2e-5, variant=variant, precision=F32)
    u = fields(n, 2, F32, shift=0.03)
    out = G.ac_fine_propagate_slices(fp, steps, u)
    assert (out.double() - field_ref(u, fp, steps)).abs().max().item() < 1.2e-7 * (steps + 1)
    if variant:
        assert (out.double().mean(dim=(1, 2)) - u.double().mean(dim=(1, 2))).abs().max().item() < 1e-8


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("n,count,steps", [(32, 3, 1), (32, 41, 4), (64, 1, 3), (64, 5, 2), (128, 1, 3), (128, 9, 2)])
def test_cube_stream(n, count, steps, variant):
    """Chunk lengths from 8 to 32 planes, in place and out of place."""
    dt = 1e-4
    fp = G.FineParams(n, float(np.sqrt(2.5e-3 / (4 * dt))) / n, 2.0, dt, variant=variant, precision=F32)
    g = torch.Generator(device="cuda").manual_seed(n + count)
    u = torch.rand((count, n, n, n), generator=g, device="cuda") * 1.8 - 0.85
    out = G.ac_fine3d_propagate(fp, steps, u)
    assert (out.double() - field_ref(u, fp, steps)).abs().max().item() < 1.2e-7 * (steps + 1)
    if variant:
        assert (out.double().mean(dim=(1, 2, 3)) - u.double().mean(dim=(1, 2, 3))).abs().max().item() < 1e-8
    v = u.clone()
    G.ac_fine3d_propagate(fp, steps, v, v)
    assert torch.equal(v, out)


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("n,prec,steps,every", [(32, F32, 7, 3), (128, F32, 9, 4), (64, F64, 11, 4), (128, F64, 6, 6), (32, F64, 5, 8)])
def test_energy_gradient_with_and_without_the_overlap(n, prec, steps, every, variant):
    """The states of a segment recomputed beside the adjoint of the next one:
    the same bits as one after the other (a workspace with one segment's room)."""
    import ctypes
    from paper_2510_07672_gb300 import abi
    fp = params(n, prec, variant, 1e-3)
    u = fields(n, 1, prec)[0]
    got = G.ac_energy_gradient_ic(fp, steps, u, checkpoint_every=every)
    p = fp.c()
    full = G.load().ac_energy_gradient_workspace(ctypes.byref(p), steps, every)
    nbytes = full - u.numel() * u.element_size() * (every + 1)
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    ref = torch.empty_like(u)
    args = (ctypes.byref(p), steps, every, u.data_ptr(), ref.data_ptr(), ws.data_ptr())
    stream = torch.cuda.current_stream().cuda_stream
    assert G.load().ac_energy_gradient_ic(*args, nbytes, stream) == abi.AC_OK
    torch.cuda.synchronize()
    assert torch.equal(got, ref)
    assert G.load().ac_energy_gradient_ic(*args, nbytes - 1, stream) == -1
