"""FP32 marches of tiny amplitude: sums below the smallest normal number keep what FP32 holds of them.

A march is linear, and a power of two scales every FP32 value exactly until denormal numbers appear.  Scaled by 2^-114,
some sums of the three weakly forced frequencies (10^-3 of the first) fall below 1.2e-38; their denormal form still
holds them to 1e-45, 10^-9 of the rows' largest entries (1e-35).  Tolerance: the FP32 parity tolerance, 2e-5, per
frequency, to the unscaled march."""
import numpy as np
import pytest

import workloads as W
from parity import rel_rows

pytestmark = pytest.mark.gpu


def test_tiny_amplitudes(rsv):
    import torch
    sysm = W.ADR2D(nx=40, ny=24, lx=40.0, ly=10.0, sponge_cells=4, visc=0.02)
    w = W.Workload("adr_tiny", sysm, np.linspace(0.0, 4.0, 4), 0.47, 2, "ssrm", n_transient_windows=2, real_state=True, seed=5)
    op = rsv.create_for_workload(w, rsv.RSV_PREC_FP32)
    try:
        x = torch.from_numpy(W.test_block(w)).to(device="cuda", dtype=torch.complex64)
        x[1:] *= 1e-3
        y, z = torch.empty_like(x), torch.empty_like(x)
        rsv.rsv_march_direct(op, x, w.k, y, **rsv.march_opts_for(w))
        rsv.rsv_march_direct(op, x * 2.0 ** -114, w.k, z, **rsv.march_opts_for(w))
        assert rel_rows(z.cpu().numpy().astype(np.complex128) * 2.0 ** 114, y.cpu().numpy().astype(np.complex128)) < 2e-5
    finally:
        rsv.rsv_destroy_operator(op)
