"""rsv_autotune tries the tiles that untuned marches take: 2 (S + 1) steps for the step form, up to a window for the
FP64 1-D jumps (S the default tile), and the default tile where the whole march is no longer than that.  A
truncated tail keeps the default tile's check points.

Tolerances: the tuned and the untuned march differ in where the tiles end, each within the parity tolerance of the
oracle (FP32 2e-5, FP64 1e-10), so twice that of each other."""
import numpy as np
import pytest

import workloads as W
from parity import rel_rows

pytestmark = pytest.mark.gpu


def _adr(steps, variant="ssrm", tail=0):
    sysm = W.ADR2D(nx=40, ny=24, lx=40.0, ly=10.0, sponge_cells=4, visc=0.02)
    return W.Workload("adr_tuned", sysm, np.linspace(0.0, 4.0, 6), 2 * np.pi / 0.8 / steps, 4, variant, n_transient_windows=0,
                      tail_steps=tail, real_state=True, seed=W.SEED_BASE + 107)


def _gl(steps):
    sysm = W.GL1D(n=(90,), mu0=(-0.2,), x0=-40.0, x1=40.0, mu2=-1e-5)
    return W.Workload("gl_tuned", sysm, np.linspace(-2.0, 2.0, 6), 2 * np.pi / 0.8 / steps, 4, "ssrm", n_transient_windows=0,
                      seed=W.SEED_BASE + 108)


@pytest.mark.parametrize("w,prec,longest", [(_adr(900), 1, 512), (_adr(256), 1, 512), (_adr(255), 1, 255), (_adr(900), 0, 256),
                                            (_gl(900), 0, 900), (_gl(900), 1, 256), (_gl(200), 0, 256)])
def test_tuned_tiles(rsv, w, prec, longest):
    import torch
    op = rsv.create_for_workload(w, prec)
    try:
        x = torch.from_numpy(W.test_block(w)).to(device="cuda", dtype=torch.complex128 if prec == 0 else torch.complex64)
        y, z = torch.empty_like(x), torch.empty_like(x)
        opts = rsv.march_opts_for(w)
        rsv.rsv_march_direct(op, x, w.k, y, **opts)
        tile, group = rsv.rsv_autotune(op, x, w.k, **opts)
        assert tile in (longest, longest // 2) and group in (4, 2, 1)
        rsv.rsv_march_direct(op, x, w.k, z, **opts)
        assert f"tile={tile} group={group}" in rsv.rsv_describe(op)
        assert rel_rows(z.cpu().numpy().astype(np.complex128), y.cpu().numpy()) < 2 * (1e-10 if prec == 0 else 2e-5)
        if w.real_state:
            trm = dict(variant="trm", tail_steps=2000, tail_tol=1e-3)
            rsv.rsv_march_direct(op, x, w.k, z, **trm)
            assert int(rsv.rsv_describe(op).split("tile=")[1].split()[0]) <= (256 if prec == 0 else 255)
    finally:
        rsv.rsv_destroy_operator(op)
