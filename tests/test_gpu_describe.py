"""rsv_describe names the kernels of the latest march: FP64 1-D marches jump up to one (instance, vector) pair per SM and
take the tile kernel above it; a sampled-forcing run of a 2-D operator takes the stage-pair kernels."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def test_1d_path_follows_the_vectors(rsv):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    sysm = W.GL1D(n=(40,), mu0=(-0.2,), x0=-20.0, x1=20.0)
    w = W.Workload("gl_path", sysm, np.linspace(-2.0, 2.0, 4), 0.05, 2, "ssrm", seed=W.SEED_BASE + 111)
    op = rsv.create_for_workload(w, rsv.RSV_PREC_FP64)
    try:
        assert "path=cuda-core jump kernels" in rsv.rsv_describe(op)
        for k, path in ((sms + 1, "path=cuda-core tile kernel"), (sms, "path=cuda-core jump kernels")):
            x = torch.ones(w.n_omega, k, w.n, dtype=torch.complex128, device="cuda")
            rsv.rsv_march_direct(op, x, k, torch.empty_like(x))
            assert path in rsv.rsv_describe(op)
    finally:
        rsv.rsv_destroy_operator(op)


def test_2d_path_follows_the_forcing(rsv):
    import torch
    sysm = W.ADR2D(nx=40, ny=24, lx=40.0, ly=10.0, sponge_cells=4, visc=0.02)
    w = W.Workload("adr_path", sysm, np.linspace(0.0, 4.0, 6), 0.4, 1, "ssrm", real_state=True, seed=W.SEED_BASE + 112)
    op = rsv.create_for_workload(w, rsv.RSV_PREC_FP32)
    try:
        f = torch.zeros(4, 1, w.n, device="cuda")
        rsv.rsv_series_march(op, False, 1, torch.zeros(6, 1, w.n, device="cuda"), 6, forcing=f, n_in=4, every=2)
        assert "path=cuda-core 2-D stage-pair kernels" in rsv.rsv_describe(op)
        x = torch.zeros(w.n_omega, 1, w.n, dtype=torch.complex64, device="cuda")
        rsv.rsv_march_direct(op, x, 1, torch.empty_like(x))
        assert "path=cuda-core 2-D step kernel" in rsv.rsv_describe(op)
    finally:
        rsv.rsv_destroy_operator(op)
