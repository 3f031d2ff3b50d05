"""A march whose step form does not fit next to other allocations runs at the stage times instead of failing.

2-D, 512 x 512, 128 frequencies, one vector, FP32: accumulators 537 MB; the step form needs 268 MB of transformed
coefficients, 64 MB of temporary, tiles of 16 steps (34 MB) and 3 MB of states on top, the stage form tiles of 55 MB.
The rest of the device is filled until 0.9 of what is free lies between the two (740 of 592 and 906 MB), then until it
lies between the stage form's and the step form's tiles of 127 steps (1000 of 941 and 1138 MB), where the tuner's
trials fit in the stage form only and the march after it in the step form with a shorter tile.  Tolerance:
both marches are within the FP32 parity tolerance of 2e-5 of the oracle, so within twice that of each other."""
import numpy as np
import pytest

import workloads as W
from parity import rel_rows

pytestmark = pytest.mark.gpu


def test_step_form_falls_back_to_stage_times(rsv):
    import torch
    sysm = W.ADR2D(nx=512, ny=512, lx=40.0, ly=10.0, sponge_cells=8)
    w = W.Workload("adr_memory", sysm, np.linspace(0.0, 40.0, 128), 0.5 * 40.0 / 513, 1, "ssrm", n_transient_windows=0,
                   real_state=True, seed=W.SEED_BASE + 109)
    gen = torch.Generator(device="cuda").manual_seed(109)
    x = torch.randn(w.n_omega, 1, w.n, dtype=torch.complex64, device="cuda", generator=gen)
    x[0].imag.zero_()
    y, z = torch.empty_like(x), torch.empty_like(x)
    opts = rsv.march_opts_for(w)
    op = rsv.create_for_workload(w, rsv.RSV_PREC_FP32)
    rsv.rsv_march_direct(op, x, 1, y, **opts)
    assert "tile=255 " in rsv.rsv_describe(op)     # 256 columns: one sum per tile
    want = y.cpu().numpy()      # compared on the host: the device is full
    rsv.rsv_destroy_operator(op)
    op = rsv.create_for_workload(w, rsv.RSV_PREC_FP32)
    filler = []
    try:
        torch.cuda.empty_cache()
        free, _ = torch.cuda.mem_get_info()
        filler.append(torch.empty(free - 822 * 10 ** 6, dtype=torch.uint8, device="cuda"))
        for _ in range(2):
            z.fill_(float("nan"))
            rsv.rsv_march_direct(op, x, 1, z, **opts)
        assert rel_rows(z.cpu().numpy(), want) < 4e-5
        filler.clear()
        torch.cuda.empty_cache()
        rsv.rsv_destroy_operator(op)
        op = rsv.create_for_workload(w, rsv.RSV_PREC_FP32)
        free, _ = torch.cuda.mem_get_info()
        filler.append(torch.empty(free - 1111 * 10 ** 6, dtype=torch.uint8, device="cuda"))
        assert rsv.rsv_autotune(op, x, 1, **opts) == (127, 1)
        rsv.rsv_march_direct(op, x, 1, z, **opts)
        assert rel_rows(z.cpu().numpy(), want) < 4e-5
    finally:
        filler.clear()
        torch.cuda.empty_cache()
        rsv.rsv_destroy_operator(op)


def test_equal_host_marches_plan_equally(rsv):
    """Host-input march of 8 vectors of 256 x 256, 64 frequencies: 3.56 GB of workspaces, 537 MB of them staging buffers.
    With 0.9 x 4.11 GB free the first march holds all 8 vectors; so does the second one, beside the buffers of the
    first, and gives the same bits."""
    import torch
    sysm = W.ADR2D(nx=256, ny=256, lx=40.0, ly=10.0, sponge_cells=8)
    w = W.Workload("adr_host_memory", sysm, np.linspace(0.0, 40.0, 64), 0.5 * 40.0 / 257, 8, "ssrm", n_transient_windows=0,
                   real_state=True, seed=W.SEED_BASE + 110)
    gen = torch.Generator().manual_seed(110)
    x = torch.randn(w.n_omega, w.k, w.n, dtype=torch.complex64, generator=gen).pin_memory()
    x[0].imag.zero_()
    y = torch.empty(x.shape, dtype=x.dtype, device="cuda")
    op = rsv.create_for_workload(w, rsv.RSV_PREC_FP32)
    filler = []
    try:
        torch.cuda.empty_cache()
        free, _ = torch.cuda.mem_get_info()
        filler.append(torch.empty(free - 4111 * 10 ** 6, dtype=torch.uint8, device="cuda"))
        outs = []
        for _ in range(2):
            rsv.rsv_march_direct_host(op, x, w.k, y, **rsv.march_opts_for(w))
            assert "group=8 " in rsv.rsv_describe(op)
            outs.append(y.cpu())
        assert torch.equal(outs[0], outs[1])
    finally:
        filler.clear()
        torch.cuda.empty_cache()
        rsv.rsv_destroy_operator(op)
