"""Small single-kernel cases for profiling with ncu.

    python -m paper_2510_07672_gb300.profile_cases fine     # ac_fine_propagate_slices, 512 x 256^2, 20 steps (stencil_reg_kernel)
    python -m paper_2510_07672_gb300.profile_cases fine_fft # the same by the Fourier solve (fine_field_kernel)
    python -m paper_2510_07672_gb300.profile_cases conv     # cnn_coarse_step, 16 x 256^2, 1-32x6-1 gelu bf16, mass shift
    python -m paper_2510_07672_gb300.profile_cases conv64   # cnn_coarse_step, 1 x 1024^2, 1-64x8-1 gelu bf16
    python -m paper_2510_07672_gb300.profile_cases big      # ac_fine_propagate_slices, 16 x 1024^2, 4 steps (big_tile_kernel)
    python -m paper_2510_07672_gb300.profile_cases big_fft  # 2 steps too stiff for the tiles (big_rows_kernel, big_cols_kernel)
    python -m paper_2510_07672_gb300.profile_cases acnn     # acnn_forward (fused), 512 x 256^2, C = 4, 2 blocks
    python -m paper_2510_07672_gb300.profile_cases fine3d   # ac_fine3d_propagate, 16 x 128^3, 2 steps (cube_kernel)
    python -m paper_2510_07672_gb300.profile_cases fine3d_fft # 1 step too stiff for the streamed planes (fine3d_pass)
    python -m paper_2510_07672_gb300.profile_cases train    # cnn forward and backward, 16 x 256^2, 1-64x3-1 (wgrad_tc_kernel)
    python -m paper_2510_07672_gb300.profile_cases acnn_train # ACNN forward and backward, 16 x 256^2, C = 4 (strip kernels)

Each case runs its call twice (a warm-up launch, then the one to capture) and
exits 0, so `ncu -s <warm-up launches> -c 1` captures a warm launch.  Inputs
are the benchmark's seeded synthetic fields.
"""
from __future__ import annotations

import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def main(case: str) -> None:
    import numpy as np
    import torch

    import acpr_inputs as I
    import paper_2510_07672_gb300 as G

    W = I.MASS_F32_256
    if case in ("fine", "fine_fft"):
        u = torch.tensor(np.stack([I.random_field(W.n, seed=s, zero_mean=True) for s in range(512)]),
                         dtype=torch.float32, device="cuda")
        fp = G.FineParams(W.n, W.eps, W.S, W.dt, variant=W.variant, precision=G.AC_F32)
        out = torch.empty_like(u)
        G.ac_fine_set_variant(W.n, G.AC_F32, 1 if case == "fine_fft" else 0)
        for _ in range(2):
            G.ac_fine_propagate_slices(fp, 20, u, out)
    elif case == "conv":
        wt, bs = W.weights()
        net = G.CoarseNet(W.layers, W.channels, wt.astype(np.float32), bs.astype(np.float32), act=W.act,
                          precision=G.AC_F32, mass_fix=W.mass_fix)
        u = torch.tensor(W.ics(), dtype=torch.float32, device="cuda")
        for _ in range(2):
            G.cnn_coarse_step(net, u)
    elif case == "conv64":
        wt, bs = I.cnn_weights(8, 64, seed=0, sigma=0.05)
        net = G.CoarseNet(8, 64, wt.astype(np.float32), bs.astype(np.float32), act=G.AC_ACT_GELU, precision=G.AC_F32)
        u = torch.tensor(I.random_field(1024, seed=0)[None], dtype=torch.float32, device="cuda")
        for _ in range(2):
            G.cnn_coarse_step(net, u)
    elif case in ("big", "big_fft"):
        n = 1024
        u = torch.tensor(np.stack([I.random_field(n, seed=s) for s in range(16)]), dtype=torch.float32,
                         device="cuda")
        stiff = case == "big_fft"
        fp = G.FineParams(n, 0.004, 2.0, 2e-4 if stiff else 2e-5, variant=G.AC_CLASSIC, precision=G.AC_F32)
        out = torch.empty_like(u)
        for _ in range(2):
            G.ac_fine_propagate_slices(fp, 2 if stiff else 4, u, out)
    elif case == "acnn":
        w, b = I.acnn_weights(4, 2, seed=0)
        net = G.Acnn(4, 2, w, b, mass_fix=1, limiter=1, precision=G.AC_F32)
        u = torch.tensor(np.stack([I.random_field(W.n, seed=s, zero_mean=True) for s in range(512)]),
                         dtype=torch.float32, device="cuda")
        out = torch.empty_like(u)
        for _ in range(2):
            net(u, out=out)
    elif case in ("fine3d", "fine3d_fft"):
        n = 128
        u = torch.tensor(np.stack([(-0.9 + 1.8 * I.uniform01(7000 + f, I.STREAM_IC, n ** 3)).reshape(n, n, n)
                                   for f in range(16)]), dtype=torch.float32, device="cuda")
        stiff = case == "fine3d_fft"
        fp = G.FineParams(n, 0.02, 2.0, 1e-3 if stiff else 1e-4, variant=G.AC_MASS_CONSERVING, precision=G.AC_F32)
        out = torch.empty_like(u)
        for _ in range(2):
            G.ac_fine3d_propagate(fp, 1 if stiff else 2, u, out)
    elif case == "train":
        wt, bs = I.cnn_weights(3, 64, seed=0, sigma=0.05)
        net = G.TrainableCoarseNet(3, 64, wt.astype(np.float32), bs.astype(np.float32), act=G.AC_ACT_GELU)
        u = torch.tensor(W.ics(), dtype=torch.float32, device="cuda")
        ws = net.new_workspace(W.n, u.shape[0])
        for _ in range(2):
            net.forward_train(u, ws)
            net.backward(u, u, ws)
    elif case == "acnn_train":
        w, b = I.acnn_weights(4, 2, seed=0)
        net = G.Acnn(4, 2, w, b, mass_fix=1, limiter=1, precision=G.AC_F32)
        u = torch.tensor(W.ics(), dtype=torch.float32, device="cuda")
        ws = net.new_workspace(W.n, u.shape[0])
        for _ in range(2):
            net.forward_train(u, ws)
            net.backward(u, u, ws)
    else:
        raise SystemExit(f"unknown case {case!r}")
    torch.cuda.synchronize()
    print(f"{case}: ok")


if __name__ == "__main__":
    main(sys.argv[1] if len(sys.argv) > 1 else "fine")
