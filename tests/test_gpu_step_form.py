"""GPU parity of the step form (forcing transformed once per march, one forcing per step) at the sizes
where its kernels can go wrong, against the oracle.

The 2-D FP32 kernel walks strips of 120 cells in x and runs of rows in y, with rows padded to four
cells; the 3-D FP32 kernels tile 64 x 12 columns of padded rows; the FP64 stages take any grid.  The
grids below sit on and beside those edges.  Tolerances are those of the march parity tests (FP32
rounding of about 6e-8 per operation through gains of up to about 30: 2e-5; FP64 1e-10).
"""
import numpy as np
import pytest

import workloads as W
from oracle import frequencies, march, operators
from parity import rel_rows

pytestmark = pytest.mark.gpu

TOL = {0: 1e-10, 1: 2e-5}


def _check(rsv, w, matrix, prec, adjoint, **opts):
    import torch
    op = rsv.create_for_workload(w, prec)
    try:
        fh = W.test_block(w).astype(np.complex64).astype(np.complex128)
        x = torch.from_numpy(fh).to(device="cuda", dtype=torch.complex128 if prec == 0 else torch.complex64)
        y = torch.full_like(x, float("nan"))
        o = dict(rsv.march_opts_for(w), **opts)
        (rsv.rsv_march_adjoint if adjoint else rsv.rsv_march_direct)(op, x, w.k, y, **o)
        g = frequencies.make_grid(w.omegas, w.dt)
        ref = march.march(matrix, g, fh, variant=w.variant, n_trans=w.n_transient_windows, tail_steps=w.tail_steps,
                          adjoint=adjoint, real_state=w.real_state)
        assert rel_rows(y.cpu().numpy().astype(np.complex128), ref) < TOL[prec]
    finally:
        rsv.rsv_destroy_operator(op)


def _adr(nx, ny, k, sponge, variant="ssrm"):
    sysm = W.ADR2D(nx=nx, ny=ny, lx=40.0, ly=10.0, sponge_cells=sponge, visc=0.01)
    return W.Workload("adr_edges", sysm, np.linspace(0.0, 4.0, 6), min(0.2, 0.5 * 40.0 / (nx + 1)), k, variant,
                      n_transient_windows=1, tail_steps=21, real_state=True, seed=W.SEED_BASE + 81)


@pytest.mark.parametrize("nx,ny,k,sponge", [(3, 3, 1, 1), (119, 5, 3, 2), (120, 9, 2, 3), (121, 8, 1, 1),
                                            (124, 17, 2, 40), (241, 33, 1, 5), (245, 4, 5, 1)])
@pytest.mark.parametrize("adjoint", [False, True])
def test_2d_strip_and_run_edges_fp32(rsv, nx, ny, k, sponge, adjoint):
    w = _adr(nx, ny, k, sponge, "trm" if nx % 2 else "ssrm")
    _check(rsv, w, operators.adr2d(w.system), 1, adjoint, tile_steps=13)


@pytest.mark.parametrize("nx,ny,sponge", [(31, 6, 2), (33, 4, 1), (64, 10, 40)])
@pytest.mark.parametrize("adjoint", [False, True])
def test_2d_stages_fp64(rsv, nx, ny, sponge, adjoint):
    """Even ny: with an odd one the middle row lies on y = 0, where the sign of r(y) is that of a rounding error."""
    w = _adr(nx, ny, 3, sponge, "trm" if nx % 2 else "ssrm")
    _check(rsv, w, operators.adr2d(w.system), 0, adjoint, tile_steps=17)


@pytest.mark.parametrize("nx,ny,nz,k", [(3, 3, 3, 1), (61, 7, 5, 2), (63, 8, 4, 1), (65, 9, 9, 2), (67, 17, 6, 1)])
@pytest.mark.parametrize("adjoint", [False, True])
def test_3d_tile_edges_fp32(rsv, nx, ny, nz, k, adjoint):
    """Widths that are not multiples of four, one cell short of, on and past the 64-cell tile; a single tile in y, ragged
    or (17) a second one."""
    sysm = W.ADV3D(nx=nx, ny=ny, nz=nz, lx=20.0, ly=10.0, lz=10.0, visc=0.02)
    w = W.Workload("adv_edges", sysm, np.array([0.2 * np.pi * j for j in range(5)]), min(0.3, 0.5 * 20.0 / (nx + 1)), k,
                   "trm" if nx % 4 == 1 else "ssrm", n_transient_windows=1, tail_steps=19, real_state=True,
                   seed=W.SEED_BASE + 82)
    _check(rsv, w, operators.adv3d(w.system), 1, adjoint, tile_steps=14)


@pytest.mark.parametrize("nx,ny,nz,k", [(63, 11, 4, 1), (64, 12, 5, 2), (65, 13, 4, 1), (33, 24, 6, 1), (5, 25, 4, 2),
                                        (132, 26, 5, 1), (133, 27, 9, 1)])
@pytest.mark.parametrize("adjoint", [False, True])
def test_3d_tile_rows_and_inner_tiles_fp32(rsv, nx, ny, nz, k, adjoint):
    """One row short of, on and past one and two tiles of 12 rows; the last two grids have a tile with no cell beside a
    wall (x from 64, y from 12: the unmasked path) and its masked neighbours."""
    sysm = W.ADV3D(nx=nx, ny=ny, nz=nz, lx=20.0, ly=10.0, lz=10.0, visc=0.02)
    w = W.Workload("adv_rows", sysm, np.array([0.2 * np.pi * j for j in range(5)]), min(0.3, 0.5 * 20.0 / (nx + 1)), k,
                   "trm" if nx % 2 else "ssrm", n_transient_windows=1, tail_steps=19, real_state=True,
                   seed=W.SEED_BASE + 116)
    _check(rsv, w, operators.adv3d(w.system), 1, adjoint, tile_steps=14)


@pytest.mark.parametrize("prec", [0, 1])
def test_padded_rows_with_weights_and_tail_rule(rsv, prec):
    """Rows padded from 41 to 44 cells: the truncated TRM tail takes its norms over the padded state, and
    host input, vector groups and weights read and write the caller's unpadded layout."""
    import torch
    w = _adr(41, 12, 3, 2, "trm")
    a = operators.adr2d(w.system)
    g = frequencies.make_grid(w.omegas, w.dt)
    cap, tol, tile = 400 * g.n_t, 1e-4, 16
    op = rsv.create_for_workload(w, prec)
    try:
        fh = W.test_block(w).astype(np.complex64).astype(np.complex128)
        x = torch.from_numpy(fh).to(device="cuda", dtype=torch.complex128 if prec == 0 else torch.complex64)
        y, yh = torch.empty_like(x), torch.empty_like(x)
        o = dict(variant="trm", tail_steps=cap, tile_steps=tile, tail_tol=tol)
        rsv.rsv_march_direct(op, x, w.k, y, **o)
        steps = int(rsv.rsv_describe(op).split("steps=")[1].split()[0])
        ref, ref_steps = march.march(a, g, fh, variant="trm", tail_steps=cap, real_state=True, tail_tol=tol,
                                     check_every=tile, return_steps=True)
        assert steps == ref_steps
        assert rel_rows(y.cpu().numpy().astype(np.complex128), ref) < TOL[prec]
        o = dict(variant="trm", tail_steps=300, tile_steps=tile)
        n = w.n
        b = np.linspace(0.5, 1.5, n)
        rsv.rsv_set_weights(op, b=b)
        rsv.rsv_march_direct(op, x, w.k, y, **o)
        rsv.rsv_march_direct_host(op, x.cpu(), w.k, yh, group_vectors=2, **o)
        assert torch.equal(y, yh)
        ref = march.march(a, g, fh * b, variant="trm", tail_steps=300, real_state=True)
        assert rel_rows(y.cpu().numpy().astype(np.complex128), ref) < TOL[prec]
    finally:
        rsv.rsv_destroy_operator(op)
