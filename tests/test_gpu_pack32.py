"""GPU parity of the FP32 1-D RK4 marches in packs, against the oracle.

The sizes sit on the edges of the layout: groups of four points, 120 points per warp, one warp and several,
the longest instance of a pack (3840 points; 3841 takes the tile kernel), one pair per pack and packs of many
pairs, tiles that end inside a window, forcing that ends inside a tile, and a truncated tail.  Tolerance:
the FP32 tolerance of the 1-D parity tests; the damping of 0.2 and more leaves no long transients that would
amplify the rounded operator."""
import numpy as np
import pytest

import workloads as W
from oracle import frequencies, march, operators
from parity import rel_rows

pytestmark = pytest.mark.gpu

TOL32 = 2e-5


def _gl(ns, dt=0.05, k=2, variant="ssrm", tail=0):
    dx = 0.7
    sysm = W.GL1D(n=ns, mu0=(-0.2,) * len(ns), x0=-0.5 * dx * (max(ns) + 1), x1=0.5 * dx * (max(ns) + 1), mu2=-1e-5)
    return W.Workload("gl_pack", sysm, np.linspace(-2.0, 2.0, 5), dt, k, variant, n_transient_windows=1,
                      tail_steps=tail, seed=W.SEED_BASE + 93)


def _run(rsv, w, adjoint, ref=True, **opts):
    import torch
    op = rsv.create_for_workload(w, rsv.RSV_PREC_FP32)
    try:
        fh = W.test_block(w).astype(np.complex64)
        x = torch.from_numpy(fh).cuda()
        y = torch.full_like(x, float("nan"))
        (rsv.rsv_march_adjoint if adjoint else rsv.rsv_march_direct)(op, x, w.k, y, **dict(rsv.march_opts_for(w), **opts))
        got = y.cpu().numpy()
        if ref:
            g = frequencies.make_grid(w.omegas, w.dt)
            want = march.march(operators.gl1d(w.system), g, fh.astype(np.complex128), variant=w.variant,
                               n_trans=w.n_transient_windows, tail_steps=w.tail_steps, adjoint=adjoint)
            assert rel_rows(got.astype(np.complex128), want) < TOL32
        return got, rsv.rsv_describe(op)
    finally:
        rsv.rsv_destroy_operator(op)


@pytest.mark.parametrize("n", [2, 3, 4, 5, 119, 120, 121, 124, 241, 3840, 3841])
@pytest.mark.parametrize("adjoint", [False, True])
def test_sizes(rsv, n, adjoint):
    _, desc = _run(rsv, _gl((n,), k=1 if n > 1000 else 3), adjoint)
    assert ("packed step kernel" in desc) == (n <= 3840)


@pytest.mark.parametrize("tile", [0, 29])
@pytest.mark.parametrize("adjoint", [False, True])
def test_many_pairs_and_groups(rsv, tile, adjoint):
    """More pairs than one wave of CTAs holds: packs; groups of 3 vectors give the same result bit for bit."""
    ns = tuple(2 + 7 * i for i in range(1, 44))
    got, desc = _run(rsv, _gl(ns, dt=0.11, k=5, variant="trm", tail=61), adjoint, tile_steps=tile)
    assert "packed=" in desc
    again, _ = _run(rsv, _gl(ns, dt=0.11, k=5, variant="trm", tail=61), adjoint, ref=False, tile_steps=tile, group_vectors=3)
    assert np.array_equal(got, again)


def test_truncated_tail(rsv):
    w = _gl((150, 31), k=2, variant="trm", tail=4000)
    got, desc = _run(rsv, w, False, tail_tol=1e-7, tile_steps=64)
    assert "steps=%d " % (4000 + frequencies.make_grid(w.omegas, w.dt).n_t) not in desc
