"""FP64 marches of a block cut into uneven vector groups: the same bits as the whole block, and the oracle's values.

The FP64 analysis splits its steps into runs whose partial sums go through a buffer.  The sizes here are those where
a smaller last group would ask for more runs than the full group if the split followed the rows of a group: one run
for the full group and two for the last one (2-D), and a buffer that the last group would overrun (1-D, a window
of 4000 steps).  Tolerance against the oracle: the FP64 parity tolerance of 1e-10."""
import numpy as np
import pytest

import workloads as W
from oracle import frequencies, march, operators
from parity import rel_rows

pytestmark = pytest.mark.gpu

TOL64 = 1e-10


def _adr(nx, ny, m, k):
    sysm = W.ADR2D(nx=nx, ny=ny, lx=40.0, ly=10.0, sponge_cells=8, visc=0.01)
    return W.Workload("adr_groups", sysm, np.linspace(0.0, 4.0, m), 0.5 * 40.0 / (nx + 1), k, "ssrm", n_transient_windows=0,
                      real_state=True, seed=W.SEED_BASE + 101)


def _gl(n, m, k, steps):
    sysm = W.GL1D(n=(n,), mu0=(-0.2,), x0=-60.0, x1=60.0, mu2=-1e-5)
    omegas = np.linspace(-1.5, 1.5, m)
    return W.Workload("gl_groups", sysm, omegas, 2 * np.pi / (omegas[1] - omegas[0]) / steps, k, "ssrm",
                      n_transient_windows=0, seed=W.SEED_BASE + 102)


@pytest.mark.parametrize("w,group", [(_adr(200, 100, 16, 3), 2), (_adr(160, 200, 8, 5), 3), (_gl(256, 32, 11, 4000), 6)])
@pytest.mark.parametrize("host", [False, True])
def test_uneven_groups(rsv, w, group, host):
    import torch
    op = rsv.create_for_workload(w, rsv.RSV_PREC_FP64)
    try:
        fh = W.test_block(w)
        x = torch.from_numpy(fh).cuda()
        whole, cut = torch.empty_like(x), torch.full_like(x, float("nan"))
        opts = rsv.march_opts_for(w)
        rsv.rsv_march_direct(op, x, w.k, whole, **opts)
        f = rsv.rsv_march_direct_host if host else rsv.rsv_march_direct
        f(op, torch.from_numpy(fh) if host else x, w.k, cut, group_vectors=group, **opts)
        assert f"group={group}" in rsv.rsv_describe(op)
        assert torch.equal(whole, cut)
        g = frequencies.make_grid(w.omegas, w.dt)
        a = operators.adr2d(w.system) if w.real_state else operators.gl1d(w.system)
        ref = march.march(a, g, fh, variant="ssrm", n_trans=0, real_state=w.real_state)
        assert rel_rows(whole.cpu().numpy(), ref) < TOL64
    finally:
        rsv.rsv_destroy_operator(op)
