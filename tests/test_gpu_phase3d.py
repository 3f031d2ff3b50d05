"""Systematic rounding of the FP32 3-D half-step march, against the FP64 march of the same operator and input.

Wave speed.  A relative error e of the advection factor h / (2 dx) turns the response at frequency w by about w L e (waves of unit
speed that have crossed up to L = 20: 55 rad at the highest frequency here), and adds up over every step.  On this grid
the factor's correctly rounded FP32 value is 1.9e-9 off, its product of rounded parts 6.2e-8 (3e-6 rad).  What is left:
1e-7 of that and U's own rounding, 3e-8 per cell, random along a path of 98 cells, 55 x 3e-8 / sqrt(98) = 1.6e-7;
tolerance 1e-6.

Long schedules.  What the rows of the rounded operator do not add up to acts as damping or growth; of the factors of a
merged x coupling 1e-8 per step is left, 1e-5 over the 972 steps below where the flow is slow.  Without that there
remain the rounding of every value to FP32 once per step and of its increment, 3.6e-8 together, a random walk of at
most sqrt(972) x 3.6e-8 = 1.1e-6; tolerance 1.2e-6 (2-norm, per frequency).

The contractions run on the CUDA cores, so that theirs is the FP32 rounding only."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _march_both(rsv, w, adjoint):
    import torch
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
    return outs


@pytest.mark.parametrize("adjoint", [False, True])
def test_long_schedule(rsv, adjoint, monkeypatch):
    monkeypatch.setenv("RSV_CONTRACT_TENSOR", "0")
    sysm = W.ADV3D(nx=96, ny=48, nz=48, lx=20.0, ly=10.0, lz=10.0, visc=5e-4)
    w = W.Workload("adv_long", sysm, 0.08 * np.pi * np.arange(4), 0.5 * 20.0 / 97, 1, "ssrm", n_transient_windows=3,
                   real_state=True, seed=W.SEED_BASE + 117)
    ref, got = _march_both(rsv, w, adjoint)
    assert (np.linalg.norm(got - ref, axis=1) / np.linalg.norm(ref, axis=1)).max() < 1.2e-6


@pytest.mark.parametrize("adjoint", [False, True])
def test_phase_of_the_fastest_wave(rsv, adjoint, monkeypatch):
    monkeypatch.setenv("RSV_CONTRACT_TENSOR", "0")
    sysm = W.ADV3D(nx=98, ny=40, nz=24, lx=20.0, ly=10.0, lz=10.0, visc=5e-4)
    w = W.Workload("adv_phase", sysm, 0.08 * np.pi * np.arange(12), 0.5 * 20.0 / 99, 1, "ssrm", n_transient_windows=0,
                   real_state=True, seed=W.SEED_BASE + 113)
    ref, got = (o[-1] for o in _march_both(rsv, w, adjoint))
    assert abs((np.vdot(ref, got) / np.vdot(ref, ref)).imag) < 1e-6
