"""Performance cases of the library: what a user of the framework has it do, through its public entry points.

Every case is a dict of plain values whose "kind" names the call:

  step      ac_fine_step                  one fine step of a few fields (the smallest call)
  slices    ac_fine_propagate_slices      the fine propagator F over a batch of slices
  work      ac_fine_propagate_work        F over a list of items of uneven step counts
  adjoint   ac_energy_gradient_ic         gradient of the final energy through a fine solve
  coarse    cnn_coarse_step               one application of the conv-stack coarse propagator G
  train     TrainableCoarseNet            one training iteration of G (unrolled MSE, backward, Adam)
  acnn      Acnn                          one update of the ResBlock network (forward, scheme-residual loss, backward, Adam)
  cube      ac_fine3d_propagate           fine steps on the periodic cube
  parareal  Parareal.solve                a whole Parareal solve

Fields are drawn as the solver meets them: the first slice of a run is the random datum U(-0.9, 0.9) per grid point, the
later ones are phase fields (smooth domains of +-1 with interfaces a few eps wide), so a batch holds both.

Step counts.  A float32 solve drifts from the 64-bit one by 1e-7 to 2e-7 a step (measured: 3e-5 after 200 steps at 256^2,
1.2e-5 after 50 at 1024^2, 2e-4 over 3200), so results of many hundred steps no longer say how exact a step is.  The float32
calls here therefore take 40 to 100 steps (the range of a slice is 50 to 400) and the long rollouts are the float64 ones.
"""
import math
import os

import numpy as np
import torch

import paper_2510_07672_gb300 as G

WEIGHTS = os.path.join(os.path.dirname(os.path.abspath(G.__file__)), "weights")
S_STAB = 2.0


def listed():
    return [
        # one step of one field: what an interactive or coupled code calls per time step; latency counts
        {"name": "step_128", "kind": "step", "n": 128, "fields": 1, "f64": False, "mass": False, "eps": 2.5 / 128, "dt": 5e-5},
        # the fine phase of 16 mass-conserving problems x 32 slices of 256^2; also 512 training trajectories to the next snapshot
        {"name": "slices_256_mass", "kind": "slices", "n": 256, "fields": 512, "steps": 100, "f64": False, "mass": True,
         "eps": 0.01, "dt": 5e-5},
        # the 512^2 part of the uneven batch: items of uneven step counts, longest first
        {"name": "work_512", "kind": "work", "n": 512, "fields": 21, "steps_min": 50, "steps": 90, "f64": False, "mass": False,
         "eps": 2.5 / 512, "dt": 5e-5},
        # the large problem's slices (a share of them, and of their steps), fields too large for one cluster
        {"name": "slices_1024", "kind": "slices", "n": 1024, "fields": 32, "steps": 50, "f64": False, "mass": False,
         "eps": 0.004, "dt": 2e-5},
        # gradient of the final energy with respect to the initial field in float64 (as its finite-difference check needs it),
        # a checkpoint every 32 steps, a last segment that is not full
        {"name": "adjoint_256_f64", "kind": "adjoint", "n": 256, "steps": 300, "every": 32, "f64": True, "mass": False,
         "eps": 0.01, "dt": 5e-5},
        # one G of the benchmark on its 16 problems (trained 1-32x6-1 GELU with the mass shift)
        {"name": "coarse_256_c32", "kind": "coarse", "n": 256, "fields": 16, "channels": 32, "layers": 6, "gelu": True,
         "mass": True, "f64": False, "weights": "mass256_c32l6_gelu"},
        # one G of the large problem (trained 1-64x8-1 GELU, one field)
        {"name": "coarse_1024_c64", "kind": "coarse", "n": 1024, "fields": 1, "channels": 64, "layers": 8, "gelu": True,
         "mass": False, "f64": False, "weights": "large1024_c64l8_gelu"},
        # one training iteration of the 1-64x8-1 network: batch 16 of 256^2, two unrolled steps
        {"name": "train_256_c64", "kind": "train", "n": 256, "fields": 16, "channels": 64, "layers": 8, "gelu": True,
         "mass": False, "unroll": 2, "eps": 0.01, "dt": 5e-5},
        # one update of Algorithm 1 on the paper's ResBlock network (C = 4, 2 blocks, mass shift and limiter)
        {"name": "acnn_update_256", "kind": "acnn", "n": 256, "fields": 16, "channels": 4, "blocks": 2, "mass": True,
         "eps": 0.01, "dt": 0.01},
        # the 3D fine step: 16 mass-conserving fields of 128^3
        {"name": "cube_128", "kind": "cube", "n": 128, "fields": 16, "steps": 20, "f64": False, "mass": True, "eps": 0.02,
         "dt": 1e-4},
        # a whole Parareal solve: the plain method in float64 (64^2, 8 slices of 100 steps, tanh conv 1-16-16-16-1)
        {"name": "parareal_64_f64", "kind": "parareal", "n": 64, "problems": 1, "slices": 8, "steps": 100, "channels": 16,
         "layers": 4, "gelu": False, "mass": False, "f64": True, "eps": 0.025, "dt": 1e-4, "tol": 1e-10, "weights": ""},
        # a whole Parareal solve of the benchmark's 16 problems (its network and grid, fewer and shorter slices), run to k = s
        {"name": "parareal_256", "kind": "parareal", "n": 256, "problems": 16, "slices": 4, "steps": 40, "channels": 32,
         "layers": 6, "gelu": True, "mass": True, "f64": False, "eps": 0.01, "dt": 5e-5, "tol": 1e-6,
         "weights": "mass256_c32l6_gelu"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _fine_sizes(rng, f64, most):
    """(n, fields, steps) within `most` cell-steps."""
    n = rng.choice((16, 32, 64, 128, 256) if f64 else (16, 32, 64, 128, 256, 512))
    steps = _log(rng, 1, 300 if f64 else 80)
    fields = _log(rng, 1, max(1, min(512, most // (n * n * steps))))
    return n, fields, max(1, min(steps, most // (n * n * fields)))


def draw(rng):
    kind = rng.choice(("step", "slices", "slices", "work", "adjoint", "coarse", "coarse", "train", "acnn", "cube", "parareal"))
    mass = rng.random() < 0.5
    if kind == "step":
        f64 = rng.random() < 0.25
        n = rng.choice((16, 32, 64, 128, 256) if f64 else (16, 32, 64, 128, 256, 512))
        return {"kind": kind, "n": n, "fields": _log(rng, 1, 24), "f64": f64, "mass": mass, "eps": 2.5 / n, "dt": 5e-5}
    if kind == "slices":
        f64 = rng.random() < 0.25
        if not f64 and rng.random() < 0.2:
            return {"kind": kind, "n": 1024, "fields": _log(rng, 1, 32), "steps": _log(rng, 2, 40), "f64": False, "mass": mass,
                    "eps": 0.004, "dt": 2e-5}
        n, fields, steps = _fine_sizes(rng, f64, 60_000_000 if f64 else 3_000_000_000)
        return {"kind": kind, "n": n, "fields": fields, "steps": steps, "f64": f64, "mass": mass, "eps": 2.5 / n, "dt": 5e-5}
    if kind == "work":
        n = rng.choice((128, 256, 512))
        return {"kind": kind, "n": n, "fields": _log(rng, 3, 40 * (512 // n)), "steps_min": _log(rng, 5, 30),
                "steps": _log(rng, 40, 80), "f64": False, "mass": False, "eps": 2.5 / n, "dt": 5e-5}
    if kind == "adjoint":
        n, f64 = rng.choice((32, 64, 128, 256)), rng.random() < 0.6
        return {"kind": kind, "n": n, "steps": _log(rng, 30, 300) if f64 else _log(rng, 10, 40), "every": rng.randint(8, 48),
                "f64": f64, "mass": mass, "eps": 2.5 / n, "dt": 5e-5}
    if kind == "coarse":
        f64 = rng.random() < 0.15
        n = rng.choice((32, 64)) if f64 else rng.choice((64, 128, 256, 256, 512, 1024))
        fields = _log(rng, 1, 8) if f64 else _log(rng, 1, max(1, min(64, (1 << 21) // (n * n))))
        return {"kind": kind, "n": n, "fields": fields, "channels": 16 if f64 else rng.choice((16, 32, 32, 64)),
                "layers": rng.randint(3, 8), "gelu": rng.random() < 0.7, "mass": mass, "f64": f64, "weights": ""}
    if kind == "train":
        n = rng.choice((128, 256))
        return {"kind": kind, "n": n, "fields": _log(rng, 2, 16), "channels": rng.choice((32, 64, 64)), "layers": rng.randint(4, 8),
                "gelu": rng.random() < 0.8, "mass": mass, "unroll": rng.randint(1, 2), "eps": 2.5 / n, "dt": 5e-5}
    if kind == "acnn":
        return {"kind": kind, "n": rng.choice((64, 128, 256)), "fields": _log(rng, 2, 16), "channels": 4,
                "blocks": rng.randint(1, 3), "mass": mass, "eps": 0.01, "dt": 0.01}
    if kind == "cube":
        n = rng.choice((32, 64, 128))
        f64 = rng.random() < 0.2
        return {"kind": kind, "n": n, "fields": _log(rng, 1, (16 if n == 128 else 48) // (4 if f64 else 1)),
                "steps": _log(rng, 2, 10 if f64 else 20), "f64": f64, "mass": mass, "eps": 2.5 / n, "dt": 1e-4}
    n = rng.choice((64, 128, 256))
    f64 = n == 64 and rng.random() < 0.5
    return {"kind": kind, "n": n, "problems": rng.randint(1, 6), "slices": rng.randint(3, 8 if f64 else 5), "steps": _log(rng, 20, 100 if f64 else 30),
            "channels": 16 if f64 else 32, "layers": rng.randint(3, 6), "gelu": not f64, "mass": mass, "f64": f64,
            "eps": 2.5 / n, "dt": 5e-5, "tol": 1e-10 if f64 else 1e-6, "weights": ""}


# ---------------------------------------------------------------- inputs --

def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1000 + stream)
    return g


def _fields(seed, count, n, eps, dtype, mass, dims=2):
    """`count` fields: random data (two of three) and phase fields (one of three); zero mean where mass is conserved."""
    shape = (count,) + (n,) * dims
    u = torch.rand(shape, generator=_gen(seed, 1), device="cuda", dtype=dtype) * 1.8 - 0.9
    axes = tuple(range(1, dims + 1))
    phase = torch.arange(count, device="cuda") % 3 == 2
    if bool(phase.any()):
        m = int(phase.sum())
        k2 = sum((torch.fft.fftfreq(n, 1.0 / n, device="cuda", dtype=dtype).reshape([-1 if a == b else 1 for b in range(dims)]) ** 2
                  for a in range(dims)))
        x = torch.randn((m,) + (n,) * dims, generator=_gen(seed, 2), device="cuda", dtype=dtype)
        x = torch.fft.ifftn(torch.fft.fftn(x, dim=axes) * torch.exp(-k2 / 32.0), dim=axes).real
        x = x / x.std(dim=axes, keepdim=True)
        u[phase] = torch.tanh(x / (16.0 * eps * math.sqrt(2.0))).to(dtype) * 0.95
    if mass:
        u = u - u.mean(dim=axes, keepdim=True)
    return u.contiguous()


def _params(c):
    return G.FineParams(c["n"], c["eps"], S_STAB, c["dt"], variant=G.AC_MASS_CONSERVING if c["mass"] else G.AC_CLASSIC,
                        precision=G.AC_F64 if c.get("f64") else G.AC_F32)


def _dtype(c):
    return torch.float64 if c.get("f64") else torch.float32


def _stack_dims(c):
    L, C = c["layers"], c["channels"]
    return [(1 if l == 0 else C, 1 if l == L - 1 else C) for l in range(L)]


def _stack_weights(c, seed):
    """The committed trained weights where the case names them (the same for every seed), else seeded ones of their size."""
    if c.get("weights"):
        z = np.load(os.path.join(WEIGHTS, c["weights"] + ".npz"))
        return torch.tensor(z["w"]), torch.tensor(z["b"])
    r = np.random.RandomState(int(seed) % (1 << 31))
    w, b = [], []
    for ci, co in _stack_dims(c):
        lim = 0.7 / math.sqrt(9.0 * ci)
        w.append(r.uniform(-lim, lim, ci * co * 9))
        b.append(r.uniform(-lim, lim, co) * 0.2)
    return torch.tensor(np.concatenate(w)).to(_dtype(c)), torch.tensor(np.concatenate(b)).to(_dtype(c))


def _acnn_weights(c, seed):
    r = np.random.RandomState(int(seed) % (1 << 31))
    w, b = [], []
    for ci, co in [(1, c["channels"])] + [(c["channels"],) * 2] * (2 * c["blocks"]) + [(c["channels"], 1)]:
        lim = 1.0 / math.sqrt(9.0 * ci)
        w.append(r.uniform(-lim, lim, ci * co * 9))
        b.append(r.uniform(-lim, lim, co))
    return torch.tensor(np.concatenate(w)).float(), torch.tensor(np.concatenate(b)).float()


def _work_steps(c):
    """Step counts of the items, longest first (the same for every seed: they are the problem, not its data)."""
    r = np.random.RandomState(c["fields"] * 1009 + c["steps"])
    return sorted((int(x) for x in r.randint(min(c["steps_min"], c["steps"]), c["steps"] + 1, c["fields"])), reverse=True)


def _moments(seed, count):
    """Adam moments of a training in progress."""
    m = torch.randn(count, generator=_gen(seed, 5), device="cuda") * 1e-3
    return m, 1e-6 * (0.5 + torch.rand(count, generator=_gen(seed, 6), device="cuda"))


T_ADAM = 100  # updates done before the timed one
LR = 1e-4


def prepare(case, seed):
    c = dict(case)
    kind, n, dt = c["kind"], c["n"], _dtype(c)
    s = {"case": c}
    if kind in ("step", "slices", "work"):
        s["fp"] = _params(c)
        s["u"] = _fields(seed, c["fields"], n, c["eps"], dt, c["mass"])
        s["out"] = torch.empty_like(s["u"])
        if kind == "work":
            s["list"] = torch.tensor([[i, i, k, 0] for i, k in enumerate(_work_steps(c))], dtype=torch.int32, device="cuda")
        elif kind == "slices":
            need = G.ac_fine_workspace_bytes(n, c["fields"], s["fp"].precision)
            s["ws"] = torch.empty(need, dtype=torch.uint8, device="cuda") if need else None
    elif kind == "adjoint":
        s["fp"] = _params(c)
        s["u"] = _fields(seed, 1, n, c["eps"], dt, c["mass"])[0]
    elif kind == "coarse":
        w, b = _stack_weights(c, seed)
        s["net"] = G.CoarseNet(c["layers"], c["channels"], w, b, act=G.AC_ACT_GELU if c["gelu"] else G.AC_ACT_TANH,
                               precision=G.AC_F64 if c["f64"] else G.AC_F32, mass_fix=int(c["mass"]))
        s["u"] = _fields(seed, c["fields"], n, 2.5 / n, dt, c["mass"])
        s["out"] = torch.empty_like(s["u"])
        s["net"].ensure_work(n, c["fields"])
    elif kind == "train":
        w, b = _stack_weights(c, seed)
        net = G.TrainableCoarseNet(c["layers"], c["channels"], w, b, act=G.AC_ACT_GELU if c["gelu"] else G.AC_ACT_TANH,
                                   mass_fix=int(c["mass"]))
        net.mw, net.vw = _moments(seed, net.w.numel())
        net.mb, net.vb = _moments(seed + 7, net.b.numel())
        net.t = T_ADAM
        k = c["unroll"]
        s["net"] = net
        s["x"] = [_fields(seed, c["fields"], n, c["eps"], dt, c["mass"])] + [torch.empty(c["fields"], n, n, device="cuda") for _ in range(k)]
        # targets: the states 20 and 40 steps on
        s["target"] = []
        for _ in range(k):
            s["target"].append(_steps64(s["target"][-1] if s["target"] else s["x"][0], c, 20).contiguous())
        s["ws"] = [net.new_workspace(n, c["fields"]) for _ in range(k)]
        s["g"] = [torch.empty(c["fields"], n, n, device="cuda") for _ in range(2)]
        s["loss"] = torch.zeros(1, dtype=torch.float64, device="cuda")
        s["scratch"] = torch.empty(64, dtype=torch.float64, device="cuda")
    elif kind == "acnn":
        w, b = _acnn_weights(c, seed)
        net = G.Acnn(c["channels"], c["blocks"], w, b, mass_fix=int(c["mass"]), limiter=1)
        net.m, net.v = _moments(seed, net.nw + net.nb)
        net.t = T_ADAM
        s["net"], s["fp"] = net, _params(c)
        s["u"] = _fields(seed, c["fields"], n, c["eps"], dt, c["mass"])
        s["out"] = torch.empty_like(s["u"])
        s["ws"] = net.new_workspace(n, c["fields"])
        s["gw"], s["gb"] = torch.empty_like(net.w), torch.empty_like(net.b)
    elif kind == "cube":
        s["fp"] = _params(c)
        s["u"] = _fields(seed, c["fields"], n, c["eps"], dt, c["mass"], dims=3)
        s["out"] = torch.empty_like(s["u"])
        need = G.load().ac_fine3d_work_bytes(n, c["fields"], s["fp"].precision)
        s["work"] = torch.empty(need, dtype=torch.uint8, device="cuda")
    elif kind == "parareal":
        w, b = _stack_weights(c, seed)
        net = G.CoarseNet(c["layers"], c["channels"], w, b, act=G.AC_ACT_GELU if c["gelu"] else G.AC_ACT_TANH,
                          precision=G.AC_F64 if c["f64"] else G.AC_F32, mass_fix=int(c["mass"]))
        s["u"] = _fields(seed, c["problems"], n, c["eps"], dt, c["mass"])
        s["net"] = net
        s["pr"] = G.Parareal(_params(c), net, s["u"], c["slices"], c["steps"])
        s["pr"].enable_graphs(True)
        s["out"] = torch.empty((c["problems"], c["slices"] + 1, n, n), dtype=dt, device="cuda")
    else:
        raise ValueError(kind)
    return s


# ------------------------------------------------------------------ run --

def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "step":
        return G.ac_fine_step(s["fp"], s["u"], s["out"])
    if kind == "slices":
        if s["ws"] is not None:
            return G.ac_fine_propagate_slices_ws(s["fp"], c["steps"], s["u"], s["out"], s["ws"])
        return G.ac_fine_propagate_slices(s["fp"], c["steps"], s["u"], s["out"])
    if kind == "work":
        return G.ac_fine_propagate_work(s["fp"], s["list"], s["u"], s["out"])
    if kind == "adjoint":
        return G.ac_energy_gradient_ic(s["fp"], c["steps"], s["u"], checkpoint_every=c["every"])
    if kind == "coarse":
        return G.cnn_coarse_step(s["net"], s["u"], s["out"])
    if kind == "train":
        net, x, k = s["net"], s["x"], c["unroll"]
        scale = 1.0 / (x[0].numel() * k)
        for j in range(k):
            net.forward_train(x[j], s["ws"][j], out=x[j + 1])
        g, other = s["g"]
        for j in reversed(range(k)):
            G.mse_loss_grad(x[j + 1], s["target"][j], scale, grad=g, grad_accumulate=j < k - 1, loss=s["loss"], scratch=s["scratch"],
                            accumulate=j < k - 1)
            net.backward(x[j], g, s["ws"][j], grad_in=other if j > 0 else None, accumulate=j < k - 1)
            g, other = other, g
        net.adam(lr=LR)
        return {"x": x[1:], "loss": s["loss"], "gw": net.gw, "gb": net.gb, "w": net.w, "b": net.b, "mw": net.mw, "vw": net.vw}
    if kind == "acnn":
        net = s["net"]
        net.forward_train(s["u"], s["ws"], out=s["out"])
        loss, g = G.loss_acn(s["fp"], s["u"], s["out"])
        net.backward(s["u"], g, s["ws"], gw=s["gw"], gb=s["gb"])
        net.adam(s["gw"], s["gb"], lr=LR)
        return {"out": s["out"], "loss": loss, "g": g, "gw": s["gw"], "gb": s["gb"], "w": net.w, "b": net.b}
    if kind == "cube":
        return G.ac_fine3d_propagate(s["fp"], c["steps"], s["u"], s["out"], s["work"])
    if kind == "parareal":
        s["pr"].reset(s["u"])
        iters, _ = s["pr"].solve(c["tol"], c["slices"], allow_unconverged=True)
        return {"U": s["pr"].trajectory(s["out"]), "iters": list(iters)}
    raise ValueError(kind)


# ----------------------------------------------------------------- work --

def _step_flops(n, dims=2):
    """Two real FFTs of n^dims at 2.5 M log2 M, and ten pointwise operations per cell."""
    return n ** dims * (5 * dims * math.log2(n) + 10)


def _conv_flops(c, cells):
    return cells * sum(2 * 9 * ci * co for ci, co in _stack_dims(c))


def work(case):
    c = dict(case)
    kind, n, e = c["kind"], c["n"], 8 if case.get("f64") else 4
    if kind == "step":
        return {"bytes": 2 * e * c["fields"] * n * n, "flops": c["fields"] * _step_flops(n)}
    if kind == "slices":
        return {"bytes": 2 * e * c["fields"] * n * n, "flops": c["fields"] * c["steps"] * _step_flops(n)}
    if kind == "work":
        return {"bytes": 2 * e * c["fields"] * n * n + 16 * c["fields"], "flops": sum(_work_steps(c)) * _step_flops(n)}
    if kind == "adjoint":  # the solve and its transposed steps
        return {"bytes": 2 * e * n * n, "flops": 2 * c["steps"] * _step_flops(n)}
    if kind == "coarse":
        cells = c["fields"] * n * n
        return {"bytes": 2 * e * cells, "flops": _conv_flops(c, cells)}
    if kind == "train":  # forward, input gradients and weight gradients; inputs and targets read, predictions and updated state written
        cells = c["fields"] * n * n
        params = sum(9 * ci * co + co for ci, co in _stack_dims(c))
        return {"bytes": 4 * cells * (1 + 2 * c["unroll"]) + 7 * 4 * params, "flops": 3 * c["unroll"] * _conv_flops(c, cells)}
    if kind == "acnn":
        cells, C = c["fields"] * n * n, c["channels"]
        return {"bytes": 4 * cells * 3, "flops": 3 * cells * 18 * (2 * C + 2 * c["blocks"] * C * C)}
    if kind == "cube":
        return {"bytes": 2 * e * c["fields"] * n ** 3, "flops": c["fields"] * c["steps"] * _step_flops(n, 3)}
    # Algorithm 2 to k = s: slice n's fine solve in iterations 1 .. n + 1, G once per slice at k = 0 and s - k times at k
    s, p = c["slices"], c["problems"]
    fine = p * c["steps"] * s * (s + 1) / 2 * _step_flops(n)
    return {"bytes": e * p * (s + 2) * n * n, "flops": fine + s * (s + 1) / 2 * _conv_flops(c, p * n * n)}


# ---------------------------------------------------------------- exact --

def _symbol(c, dims=2, dtype=torch.float64):
    """(1 + S dt) + dt eps^2 mu of the periodic stencil Laplacian on the half spectrum."""
    n = c["n"]
    mu = 4.0 * n * n * torch.sin(torch.pi * torch.arange(n, device="cuda", dtype=torch.float64) / n) ** 2
    total = 0.0
    for a in range(dims):
        m = mu[: n // 2 + 1] if a == dims - 1 else mu
        total = total + m.reshape([-1 if a == b else 1 for b in range(dims)])
    return (1.0 + S_STAB * c["dt"] + c["dt"] * c["eps"] ** 2 * total).to(dtype)


def _step64(u, c, sym, dims=2):
    axes = tuple(range(-dims, 0))
    f = u - u * u * u
    if c["mass"]:
        f = f - f.mean(dim=axes, keepdim=True)
    r = (1.0 + S_STAB * c["dt"]) * u + c["dt"] * f
    return torch.fft.irfftn(torch.fft.rfftn(r, dim=axes) / sym, s=u.shape[-dims:], dim=axes)


def _steps64(u, c, steps, dims=2):
    """`steps` steps in 64 bits, a bounded number of cells at a time; the result in u's type."""
    sym, out = _symbol(c, dims), torch.empty_like(u)
    chunk = max(1, (1 << 26) // u[0].numel())
    for i in range(0, u.shape[0], chunk):
        v = u[i:i + chunk].double()
        for _ in range(steps):
            v = _step64(v, c, sym, dims)
        out[i:i + chunk] = v
    return out


def _stack64(u, w, b, c):
    x, ow, ob = u[:, None], 0, 0
    dims = _stack_dims(c)
    for l, (ci, co) in enumerate(dims):
        x = torch.nn.functional.pad(x, (1, 1, 1, 1), mode="circular")
        x = torch.nn.functional.conv2d(x, w[ow:ow + 9 * ci * co].reshape(co, ci, 3, 3), b[ob:ob + co])
        ow, ob = ow + 9 * ci * co, ob + co
        if l < len(dims) - 1:
            x = torch.nn.functional.gelu(x) if c["gelu"] else torch.tanh(x)
    x = x[:, 0]
    if c["mass"]:
        x = x - x.mean(dim=(1, 2), keepdim=True)
    return u + x


def _adam64(p, g, m, v, t):
    m1, v1 = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
    return p - LR * (m1 / (1 - 0.9 ** t)) / (torch.sqrt(v1 / (1 - 0.999 ** t)) + 1e-8), m1, v1


def _exact_train(c, seed):
    s = prepare(c, seed)
    net = s["net"]
    par = [t.double().clone().requires_grad_(True) for t in (net.w, net.b)]
    mom = [t.double() for t in (net.mw, net.vw, net.mb, net.vb)]
    x0, target, k = s["x"][0], [t.double() for t in s["target"]], c["unroll"]
    del s, net
    scale = 1.0 / (x0.numel() * k)
    loss, xs = 0.0, [torch.empty(x0.shape, dtype=torch.float64, device="cuda") for _ in range(k)]
    chunk = max(1, (1 << 17) // (c["n"] * c["n"]))
    for i in range(0, x0.shape[0], chunk):
        x, part = x0[i:i + chunk].double(), 0.0
        for j in range(k):
            x = _stack64(x, *par, c)
            xs[j][i:i + chunk] = x.detach()
            part = part + scale * ((x - target[j][i:i + chunk]) ** 2).sum()
        part.backward()
        loss = loss + part.detach()
    w, mw, vw = _adam64(par[0].detach(), par[0].grad, mom[0], mom[1], T_ADAM + 1)
    b, _, _ = _adam64(par[1].detach(), par[1].grad, mom[2], mom[3], T_ADAM + 1)
    # with the mass shift the bias gradients nearly cancel: what is left of them is the rounding of the 16-bit operands
    return {"x": xs, "loss": loss.reshape(1), "gw": par[0].grad, "gb": None if c["mass"] else par[1].grad, "w": w, "b": b, "mw": mw, "vw": vw}


def _exact_acnn(c, seed):
    s = prepare(c, seed)
    net, n, C = s["net"], c["n"], c["channels"]
    w, b = (t.double().clone().requires_grad_(True) for t in (net.w, net.b))
    m, v, u = net.m.double(), net.v.double(), s["u"].double()
    off = [0, 0]

    def conv(x, ci, co):
        ow, ob = off
        off[0], off[1] = ow + 9 * ci * co, ob + co
        x = torch.nn.functional.pad(x, (1, 1, 1, 1), mode="circular")
        return torch.nn.functional.conv2d(x, w[ow:ow + 9 * ci * co].reshape(co, ci, 3, 3), b[ob:ob + co])

    x = torch.tanh(conv(u[:, None], 1, C))
    for _ in range(c["blocks"]):
        y = torch.tanh(conv(x, C, C))
        x = x + torch.tanh(conv(y, C, C))
    x = conv(x, C, 1)[:, 0]
    if c["mass"]:
        x = x + u.mean(dim=(1, 2), keepdim=True) - x.mean(dim=(1, 2), keepdim=True)
    out = x.clamp(-1.0, 1.0)
    out.retain_grad()

    def rhs(z):
        lap = n * n * (z.roll(1, 1) + z.roll(-1, 1) + z.roll(1, 2) + z.roll(-1, 2) - 4 * z)
        f = z - z * z * z
        return c["eps"] ** 2 * lap + f - (f.mean(dim=(1, 2), keepdim=True) if c["mass"] else 0.0)

    loss = ((out - u - 0.5 * c["dt"] * (rhs(out) + rhs(u))) ** 2).mean()
    loss.backward()
    nw = w.numel()
    w1, _, _ = _adam64(w.detach(), w.grad, m[:nw], v[:nw], T_ADAM + 1)
    b1, _, _ = _adam64(b.detach(), b.grad, m[nw:], v[nw:], T_ADAM + 1)
    return {"out": out.detach(), "loss": loss.detach().reshape(1), "g": out.grad, "gw": w.grad, "gb": b.grad, "w": w1, "b": b1}


def _exact_adjoint(c, seed):
    n, steps = c["n"], c["steps"]
    u = _fields(seed, 1, n, c["eps"], _dtype(c), c["mass"])[0].double()
    sym = _symbol(c)
    states = [u]
    for _ in range(steps):
        states.append(_step64(states[-1], c, sym))
    z = states[-1]
    lap = n * n * (z.roll(1, 0) + z.roll(-1, 0) + z.roll(1, 1) + z.roll(-1, 1) - 4 * z)
    lam = (-(c["eps"] ** 2) * lap - (z - z * z * z)) / (n * n)
    for z in reversed(states[:-1]):
        mu = torch.fft.irfft2(torch.fft.rfft2(lam) / sym, s=(n, n))
        lam = (1.0 + S_STAB * c["dt"]) * mu + c["dt"] * (1.0 - 3.0 * z * z) * (mu - (mu.mean() if c["mass"] else 0.0))
    return lam


def exact(case, seed):
    c = dict(case)
    kind = c["kind"]
    if kind in ("step", "slices"):
        u = _fields(seed, c["fields"], c["n"], c["eps"], _dtype(c), c["mass"])
        return _steps64(u.double(), c, 1 if kind == "step" else c["steps"])
    if kind == "work":
        u = _fields(seed, c["fields"], c["n"], c["eps"], _dtype(c), c["mass"]).double()
        out, sym, k = torch.empty_like(u), _symbol(c), _work_steps(c)
        v, done, alive = u, 0, len(k)
        while alive:  # items are sorted: the shortest are last
            for _ in range(k[alive - 1] - done):
                v = _step64(v, c, sym)
            done = k[alive - 1]
            first = next(i for i in range(alive) if k[i] == done)
            out[first:alive] = v[first:alive]
            v, alive = v[:first], first
        return out
    if kind == "adjoint":
        return _exact_adjoint(c, seed)
    if kind == "coarse":
        w, b = (t.double().cuda() for t in _stack_weights(c, seed))
        u = _fields(seed, c["fields"], c["n"], 2.5 / c["n"], _dtype(c), c["mass"]).double()
        chunk = max(1, (1 << 19) // (c["n"] * c["n"]))
        with torch.no_grad():
            return torch.cat([_stack64(u[i:i + chunk], w, b, c) for i in range(0, u.shape[0], chunk)])
    if kind == "train":
        return _exact_train(c, seed)
    if kind == "acnn":
        return _exact_acnn(c, seed)
    if kind == "cube":
        u = _fields(seed, c["fields"], c["n"], c["eps"], _dtype(c), c["mass"], dims=3)
        return _steps64(u.double(), c, c["steps"], dims=3)
    # k = s: the trajectory is the sequential fine solve
    u = _fields(seed, c["problems"], c["n"], c["eps"], _dtype(c), c["mass"]).double()
    traj = [u]
    for _ in range(c["slices"]):
        traj.append(_steps64(traj[-1], c, c["steps"]))
    return {"U": torch.stack(traj, dim=1), "iters": None}
