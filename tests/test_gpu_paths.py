"""GPU parity at the edges of the dispatch rules of the contraction, the Gram matrix, the CUDA-core dense step
and the sampled-forcing kernels.

Contraction: 2 x 48 columns are the last with the converted operand in tensor memory, 2 x 64 the last that are
analysed in two sums per tile; windows of more than one 512-step tile.  Gram: 4 x 4 tiles of pairs (k = 4, 5,
16, 17), slabs of 256 points (255, 256, 257) and CTAs of 8192 (8193).  Dense: two chunks of K (n > 512 in FP32,
n > 256 in FP64).  Sampled forcing: tiles of 32 rows (many) and of 8 (few), against the single stages.

Tolerances: FP32 marches 2e-5 of the oracle (FP32 rounding of the state and of the synthesised forcing over some
hundred steps, as in the other FP32 parity tests; measured errors of such marches are a few 1e-6).  FP32 QR: Q
carries one rounding of X R^-1 per pass, cond(X) ~ 3, 32 terms: 32 x 6e-8 x 3 = 6e-6, R likewise.  Sampled
forcing: both paths are RK4 in FP32 with different roundings, 2e-5."""
import numpy as np
import pytest

import workloads as W
from oracle import frequencies, march, operators
from parity import rel_rows

pytestmark = pytest.mark.gpu

TOL32 = 2e-5


def _check(rsv, w, matrix, prec=1, dense=None):
    import torch
    op = rsv.create_for_workload(w, prec, **({"dense_matrix": dense} if dense is not None else {}))
    try:
        fh = W.test_block(w)
        if prec == 1:
            fh = fh.astype(np.complex64)
        x = torch.from_numpy(fh).cuda()
        y = torch.full_like(x, float("nan"))
        rsv.rsv_march_direct(op, x, w.k, y, **rsv.march_opts_for(w))
        g = frequencies.make_grid(w.omegas, w.dt)
        ref = march.march(matrix, g, fh.astype(np.complex128), variant=w.variant, n_trans=w.n_transient_windows,
                          tail_steps=w.tail_steps, real_state=w.real_state)
        assert rel_rows(y.cpu().numpy().astype(np.complex128), ref) < (TOL32 if prec == 1 else 1e-10)
        return rsv.rsv_describe(op)
    finally:
        rsv.rsv_destroy_operator(op)


@pytest.mark.parametrize("m", [48, 49, 64, 65])
def test_contraction_columns_real(rsv, m):
    sysm = W.ADR2D(nx=37, ny=12, lx=40.0, ly=10.0, sponge_cells=3, visc=0.02)
    w = W.Workload("adr_cols", sysm, 0.1 * np.arange(m), 0.11, 2, "ssrm", n_transient_windows=1, real_state=True,
                   seed=W.SEED_BASE + 95)
    assert ("tile=512" in _check(rsv, w, operators.adr2d(sysm))) == (m <= 64)


@pytest.mark.parametrize("m", [48, 49, 65])
def test_contraction_columns_complex(rsv, m):
    sysm = W.GL1D(n=(60, 31), mu0=(-0.2, -0.2), x0=-21.0, x1=21.0, mu2=-1e-5)
    w = W.Workload("gl_cols", sysm, 0.2 * (np.arange(m) - m // 2), 0.05, 3, "ssrm", n_transient_windows=1,
                   seed=W.SEED_BASE + 96)
    assert ("tile=256" in _check(rsv, w, operators.gl1d(sysm))) == (m <= 64)


@pytest.mark.parametrize("k,sizes", [(1, (8193,)), (4, (255, 256, 257)), (5, (8190,)), (16, (300, 33)), (17, (512, 64))])
def test_orthonormalize_fp32(rsv, k, sizes):
    import torch
    if sizes[0] > 4096:   # longer than a 1-D instance may be: a 2-D system of as many points
        nx = 3 if sizes[0] % 3 == 0 else 91
        sysm = W.ADR2D(nx=nx, ny=sizes[0] // nx, lx=40.0, ly=10.0, sponge_cells=1)
        sizes = (nx * (sizes[0] // nx),)
    else:
        sysm = W.GL1D(n=sizes, mu0=(-0.1,) * len(sizes), x0=-20.0, x1=20.0)
    w = W.Workload("qr32", sysm, np.linspace(0.0, 2.0, 3), 0.01, k, "ssrm", real_state=isinstance(sysm, W.ADR2D),
                   seed=W.SEED_BASE + 97)
    op = rsv.create_for_workload(w, 1)
    try:
        x = W.test_block(w).astype(np.complex64)
        xd = torch.from_numpy(x.copy()).cuda()
        r = np.zeros((w.n_omega, len(sizes), k, k), dtype=np.complex128)
        rsv.rsv_orthonormalize(op, xd, k, r)
        q = xd.cpu().numpy().astype(np.complex128)
        for j in range(w.n_omega):
            off = 0
            for i, n in enumerate(sizes):
                a = x[j, :, off:off + n].astype(np.complex128).T
                qq = q[j, :, off:off + n].T
                off += n
                assert np.abs(qq.conj().T @ qq - np.eye(k)).max() < 6e-6
                assert np.abs(qq @ r[j, i] - a).max() < 6e-6 * np.abs(a).max()
    finally:
        rsv.rsv_destroy_operator(op)


@pytest.mark.parametrize("n,prec,k", [(520, 1, 3), (640, 1, 2), (260, 0, 2)])
def test_dense_step_in_two_chunks(rsv, n, prec, k):
    sysm = W.Dense(n=n, x_half_width=0.16 * n)
    w = W.Workload("dense_chunks", sysm, np.linspace(-4.0, 4.0, 5), 0.005, k, "trm", tail_steps=60)
    a = W.hermite_gl_matrix(sysm)
    assert "cuda-core propagator step" in _check(rsv, w, a, prec, a)


@pytest.mark.parametrize("nx,ny,k", [(256, 320, 8), (64, 9, 1), (132, 40, 2)])
@pytest.mark.parametrize("every", [1, 3, 9])
def test_sampled_forcing_tiles(rsv, nx, ny, k, every, monkeypatch):
    import torch
    sysm = W.ADR2D(nx=nx, ny=ny, lx=40.0, ly=10.0, sponge_cells=4, visc=0.01)
    w = W.Workload("adr_tiles", sysm, np.linspace(0.0, 4.0, 4), 0.25 * min(40.0 / (nx + 1), 10.0 / (ny + 1)), k, "trm",
                   real_state=True, seed=W.SEED_BASE + 98)
    rng = np.random.default_rng(98)
    f = torch.from_numpy(rng.standard_normal((14, k, nx * ny)).astype(np.float32)).cuda()
    outs = []
    for staged in ("0", "1"):
        monkeypatch.setenv("RSV_STENCIL2D_STAGED", staged)
        op = rsv.create_for_workload(w, 1)
        try:
            out = torch.zeros((20, k, nx * ny), dtype=torch.float32, device="cuda")
            n_out, _ = rsv.rsv_series_march(op, False, k, out, 20, forcing=f, n_in=14, every=every)
            outs.append(out[:n_out].cpu().numpy())
        finally:
            rsv.rsv_destroy_operator(op)
    assert outs[0].shape == outs[1].shape and outs[0].shape[0] >= 14
    assert np.abs(outs[0] - outs[1]).max() < 2e-5 * np.abs(outs[1]).max()
