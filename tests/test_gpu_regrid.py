"""One operator on two frequency grids: the second grid has another step h, the same vectors, tile length and
workspaces.  Its marches give the bits that a fresh operator gives, although tiles of the first grid were captured
into graphs."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _adr():
    sysm = W.ADR2D(nx=40, ny=24, lx=40.0, ly=10.0, sponge_cells=4)
    return W.Workload("adr_regrid", sysm, np.linspace(0.0, 4.0, 8), 0.5 * sysm.lx / 41, 2, "ssrm", n_transient_windows=2,
                      real_state=True, seed=W.SEED_BASE + 105)


def _adv():
    sysm = W.ADV3D(nx=12, ny=8, nz=6, lx=20.0, ly=10.0, lz=10.0, visc=0.02)
    return W.Workload("adv_regrid", sysm, np.linspace(0.0, 4.0, 8), 0.5 * sysm.lx / 13, 2, "ssrm", n_transient_windows=2,
                      real_state=True, seed=W.SEED_BASE + 106)


@pytest.mark.parametrize("make", [_adr, _adv])
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("adjoint", [False, True])
def test_second_grid_after_graphs(rsv, make, prec, adjoint):
    import torch
    w = make()
    x = torch.from_numpy(W.test_block(w)).to(device="cuda", dtype=torch.complex128 if prec == 0 else torch.complex64)
    march = rsv.rsv_march_adjoint if adjoint else rsv.rsv_march_direct
    second = np.linspace(0.0, 3.5, 8)
    got, want = torch.empty_like(x), torch.empty_like(x)
    op, fresh = rsv.create_for_workload(w, prec), rsv.create_for_workload(w, prec)
    try:
        opts = rsv.march_opts_for(w, tile_steps=7)
        for _ in range(2):
            march(op, x, w.k, got, **opts)
        assert int(rsv.rsv_describe(op).split("graphs=")[1].split()[0]) > 0
        _, h0 = rsv.rsv_set_frequencies(op, w.omegas)
        _, h1 = rsv.rsv_set_frequencies(op, second)
        assert h0 != h1
        rsv.rsv_set_frequencies(fresh, second)
        march(op, x, w.k, got, **opts)
        march(fresh, x, w.k, want, **opts)
        assert torch.equal(got, want)
    finally:
        rsv.rsv_destroy_operator(op)
        rsv.rsv_destroy_operator(fresh)
