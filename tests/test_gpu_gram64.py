"""FP64 QR at the widths where the Gram kernel's slabs change, k = 28 (256 points) and 29 to 32 (128 points), on
instances that end on and beside a slab and past a chunk of 2048 points.

Tolerance: Q carries one FP64 rounding of X R^-1 per pass, 32 terms, cond(X) below 10 for Gaussian columns of twice
their number and more: 2 x 32 x 1.1e-16 x 10 = 7e-14; 1e-12 with a margin for the sums over the points."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

TOL = 1e-12


@pytest.mark.parametrize("k", [1, 27, 28, 29, 31, 32])
@pytest.mark.parametrize("sizes", [(127, 128, 129), (256, 2049)])
def test_orthonormalize_fp64(rsv, k, sizes):
    import torch
    sysm = W.GL1D(n=sizes, mu0=(-0.1,) * len(sizes), x0=-20.0, x1=20.0)
    w = W.Workload("qr64", sysm, np.linspace(0.0, 2.0, 3), 0.01, k, "ssrm", seed=W.SEED_BASE + 103)
    op = rsv.create_for_workload(w, rsv.RSV_PREC_FP64)
    try:
        x = W.test_block(w)
        xd = torch.from_numpy(x.copy()).cuda()
        r = np.zeros((w.n_omega, len(sizes), k, k), dtype=np.complex128)
        rsv.rsv_orthonormalize(op, xd, k, r)
        q = xd.cpu().numpy()
        for j in range(w.n_omega):
            off = 0
            for i, n in enumerate(sizes):
                a, qq = x[j, :, off:off + n].T, q[j, :, off:off + n].T
                off += n
                assert np.abs(qq.conj().T @ qq - np.eye(k)).max() < TOL
                assert np.abs(qq @ r[j, i] - a).max() < TOL * np.abs(a).max()
                assert np.abs(np.tril(r[j, i], -1)).max() == 0 and (np.diag(r[j, i]).real > 0).all()
    finally:
        rsv.rsv_destroy_operator(op)
