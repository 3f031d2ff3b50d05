"""Wave speed of the FP32 3-D half-step march, against the FP64 march of the same operator and input.

A relative error e of the advection factor h / (2 dx) turns the response at frequency w by about w L e (waves of unit
speed that have crossed up to L = 20: 55 rad at the highest frequency here), and adds up over every step.  On this grid
the factor's correctly rounded FP32 value is 1.9e-9 off, its product of rounded parts 6.2e-8 (3e-6 rad).  What is left:
1e-7 of that and U's own rounding, 3e-8 per cell, random along a path of 98 cells, 55 x 3e-8 / sqrt(98) = 1.6e-7;
tolerance 1e-6.  The contractions run on the CUDA cores, so that theirs is the FP32 rounding only (real part)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("adjoint", [False, True])
def test_phase_of_the_fastest_wave(rsv, adjoint, monkeypatch):
    import torch
    monkeypatch.setenv("RSV_CONTRACT_TENSOR", "0")
    sysm = W.ADV3D(nx=98, ny=40, nz=24, lx=20.0, ly=10.0, lz=10.0, visc=5e-4)
    w = W.Workload("adv_phase", sysm, 0.08 * np.pi * np.arange(12), 0.5 * 20.0 / 99, 1, "ssrm", n_transient_windows=0,
                   real_state=True, seed=W.SEED_BASE + 113)
    x = torch.from_numpy(W.test_block(w)).cuda()
    outs = []
    for prec, ct in ((rsv.RSV_PREC_FP64, torch.complex128), (rsv.RSV_PREC_FP32, torch.complex64)):
        op = rsv.create_for_workload(w, prec)
        try:
            xi = x.to(torch.complex64).to(ct)
            y = torch.empty_like(xi)
            (rsv.rsv_march_adjoint if adjoint else rsv.rsv_march_direct)(op, xi, w.k, y, **rsv.march_opts_for(w))
            outs.append(y.cpu().numpy().astype(np.complex128).reshape(w.n_omega, -1))
        finally:
            rsv.rsv_destroy_operator(op)
    ref, got = outs[0][-1], outs[1][-1]
    assert abs((np.vdot(ref, got) / np.vdot(ref, ref)).imag) < 1e-6
