"""GPU parity of the FP64 1-D marches that jump over several steps, against the oracle at 1e-10.

The sizes sit on the edges of the jumps' layout: instances of one CTA, of clusters of 4 and 16 (8 where 16
do not fit), the smallest and the longest (1024 points; 1025 takes the tile kernel), steps near the
stability limit (the band of the step matrix is full) and small ones (it is cut), windows and tails that are
no multiple of the jump, Crank-Nicolson with real and complex coefficients, and a Crank-Nicolson matrix that
is not dominated by its diagonal (no jumps)."""
import numpy as np
import pytest

import workloads as W
from oracle import frequencies, march, operators
from parity import rel_rows

pytestmark = pytest.mark.gpu

TOL64 = 1e-10


def _run(rsv, w, adjoint, scheme="rk4", **opts):
    import torch
    op = rsv.create_for_workload(w, rsv.RSV_PREC_FP64, scheme=rsv.RSV_SCHEME_CN if scheme == "cn" else rsv.RSV_SCHEME_RK4)
    try:
        fh = W.test_block(w)
        x = torch.from_numpy(fh).cuda()
        y = torch.full_like(x, float("nan"))
        (rsv.rsv_march_adjoint if adjoint else rsv.rsv_march_direct)(op, x, w.k, y, **dict(rsv.march_opts_for(w), **opts))
        g = frequencies.make_grid(w.omegas, w.dt)
        ref = march.march(operators.gl1d(w.system), g, fh, variant=w.variant, n_trans=w.n_transient_windows,
                          tail_steps=w.tail_steps, adjoint=adjoint, scheme=scheme)
        assert rel_rows(y.cpu().numpy(), ref) < TOL64
        return rsv.rsv_describe(op)
    finally:
        rsv.rsv_destroy_operator(op)


def _gl(n, x_half, dt, k=2, variant="ssrm", m=5, tail=0, nu=2.0 + 0.4j):
    ns = n if isinstance(n, tuple) else (n,)
    sysm = W.GL1D(n=ns, mu0=(-0.2,) * len(ns), x0=-x_half, x1=x_half, mu2=-1e-5, nu=nu)
    return W.Workload("gl_jump", sysm, np.linspace(-2.0, 2.0, m), dt, k, variant, n_transient_windows=1,
                      tail_steps=tail, seed=W.SEED_BASE + 91)


@pytest.mark.parametrize("n", [2, 3, 31, 63, 64, 127, 128, 255, 600, 1024, 1025])
@pytest.mark.parametrize("adjoint", [False, True])
def test_sizes(rsv, n, adjoint):
    dx = 0.7
    desc = _run(rsv, _gl(n, 0.5 * dx * (n + 1), 0.11 if n % 2 else 0.02, k=1 if n > 600 else 3), adjoint)
    assert ("jump" in desc) == (n <= 1024)


@pytest.mark.parametrize("dt", [0.2, 0.05, 0.004])
@pytest.mark.parametrize("tile", [0, 29, 64])
def test_bands_and_tiles_trm(rsv, dt, tile):
    """Step factors 4 |gamma| h / dx^2 from 2.3 (full bands) to 0.05; a forcing window and a tail that are no
    multiples of the jump, tiles shorter than it and across the end of the forcing."""
    w = _gl(150, 0.5 * 0.7 * 151, dt, variant="trm", tail=101)
    _run(rsv, w, tile == 29, tile_steps=tile)


@pytest.mark.parametrize("adjoint", [False, True])
def test_uneven_instances(rsv, adjoint):
    _run(rsv, _gl((2, 140, 33, 7), 30.0, 0.05, k=4), adjoint)


@pytest.mark.parametrize("n,k", [(40, 3), (130, 2), (500, 4)])
@pytest.mark.parametrize("adjoint", [False, True])
def test_crank_nicolson(rsv, n, k, adjoint):
    w = W.gl_paper(n=n, n_omega=7, dt=0.02)
    w = W.Workload("gl_cn", w.system, w.omegas, w.dt, k, "trm" if n == 130 else "ssrm", n_transient_windows=1, tail_steps=77,
                   seed=W.SEED_BASE + 92)
    assert "jump" in _run(rsv, w, adjoint, scheme="cn")


@pytest.mark.parametrize("dt,jumps", [(0.05, True), (0.8, False)])
def test_crank_nicolson_complex(rsv, dt, jumps):
    """Strong advection: with the long step the off-diagonal couplings outweigh the diagonal."""
    w = _gl(90, 40.0, dt, k=2, nu=8.0 + 0.4j)
    assert ("jump" in _run(rsv, w, False, scheme="cn")) == jumps


def test_grouping_is_bit_exact_across_cluster_sizes(rsv):
    """Groups of 10 vectors take 8-CTA clusters, groups of 3 take 16: the same sums in the same order."""
    import torch
    w = _gl(256, 60.0, 0.02, k=10)
    op = rsv.create_for_workload(w, rsv.RSV_PREC_FP64)
    try:
        x = torch.from_numpy(W.test_block(w)).cuda()
        y, z = torch.empty_like(x), torch.empty_like(x)
        rsv.rsv_march_direct(op, x, w.k, y, **rsv.march_opts_for(w))
        rsv.rsv_march_direct(op, x, w.k, z, group_vectors=3, **rsv.march_opts_for(w))
        assert torch.equal(y, z)
    finally:
        rsv.rsv_destroy_operator(op)
