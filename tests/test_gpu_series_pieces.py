"""Sampled forcing with sample spacings that are longer than a time tile or no multiple of the 16 stage times a thread
takes.  Against the oracle at the parity tolerances (FP64 1e-10, FP32 2e-5); and the cost of a step must not grow with
the spacing (only the pieces that hold stage times of the tile are launched: the same work per step, so a factor of
three is far outside the noise, while launching every piece of an interval costs ten times more here)."""
import time

import numpy as np
import pytest

import workloads as W
from oracle import operators, series

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("every", [7, 8, 9, 40, 150, 301])
@pytest.mark.parametrize("interp", ["c0", "c2"])
def test_long_spacings(rsv, prec, every, interp):
    import torch
    sysm = W.GL1D(n=(30,), mu0=(-0.2,), x0=-15.0, x1=15.0)
    w = W.Workload("gl_pieces", sysm, np.linspace(-1.0, 1.0, 5), 0.02, 2, "ssrm", seed=W.SEED_BASE + 114)
    op = rsv.create_for_workload(w, prec)
    try:
        _, h = rsv.rsv_set_frequencies(op, w.omegas)
        ct = torch.complex128 if prec == 0 else torch.complex64
        rng = np.random.default_rng(114)
        f = rng.standard_normal((4, 2, w.n)) + 1j * rng.standard_normal((4, 2, w.n))
        fd = torch.from_numpy(f).to("cuda", ct)
        out = torch.zeros((6, 2, w.n), dtype=ct, device="cuda")
        rsv.rsv_series_march(op, False, 2, out, 6, forcing=fd, n_in=4, every=every, interp=interp)
        ref = series.series_march(operators.gl1d(sysm), h, every, 6, init=None, forcing=fd.cpu().numpy().astype(np.complex128),
                                  kind=interp, adjoint=False, scheme="rk4")
        assert np.abs(out.cpu().numpy() - ref).max() / np.abs(ref).max() < (1e-10 if prec == 0 else 2e-5)
    finally:
        rsv.rsv_destroy_operator(op)


def test_step_cost_does_not_follow_the_spacing(rsv):
    import torch
    sysm = W.ADR2D(nx=256, ny=128, lx=40.0, ly=10.0, sponge_cells=32, visc=1e-3)
    w = W.Workload("adr_pieces", sysm, np.linspace(0.0, 4.0, 8), 0.5 * 40.0 / 257, 4, "ssrm", real_state=True,
                   seed=W.SEED_BASE + 115)
    op = rsv.create_for_workload(w, 1)
    try:
        f = torch.randn(2, 4, w.n, device="cuda")
        out = torch.zeros(2, 4, w.n, device="cuda")
        cost = {}
        for every in (2000, 2000, 200000):   # the first one warms up
            torch.cuda.synchronize()
            t = time.perf_counter()
            rsv.rsv_series_march(op, False, 4, out, 2, forcing=f, n_in=2, every=every)
            torch.cuda.synchronize()
            cost[every] = (time.perf_counter() - t) / every
        assert cost[200000] < 3 * cost[2000]
    finally:
        rsv.rsv_destroy_operator(op)
