"""A frequency grid whose tables do not fit the device leaves the operator without frequencies: the call reports OOM, a
march after it RSV_ERR_STATE, and a grid that fits sets the operator up again."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def test_tables_that_do_not_fit(rsv):
    import torch
    sysm = W.GL1D(n=(40,), mu0=(-0.2,), x0=-20.0, x1=20.0)
    w = W.Workload("gl_oom", sysm, np.linspace(-2.0, 2.0, 4), 0.05, 2, "ssrm", seed=W.SEED_BASE + 118)
    op = rsv.create_for_workload(w, rsv.RSV_PREC_FP32)
    filler = []
    try:
        x = torch.from_numpy(W.test_block(w)).to("cuda", torch.complex64)
        y, z = torch.empty_like(x), torch.empty_like(x)
        rsv.rsv_march_direct(op, x, w.k, y, **rsv.march_opts_for(w))
        torch.cuda.empty_cache()
        free, _ = torch.cuda.mem_get_info()
        filler.append(torch.empty(free - 200 * 10 ** 6, dtype=torch.uint8, device="cuda"))
        dw = 2 * np.pi / (0.05 * 1.2e7)                    # 1.2e7 steps per window: a table of 384 MB
        with pytest.raises(rsv.RsvError) as e:
            rsv.rsv_set_frequencies(op, dw * np.arange(4.0))
        assert e.value.status == 6
        with pytest.raises(rsv.RsvError) as e:
            rsv.rsv_march_direct(op, x, w.k, z, **rsv.march_opts_for(w))
        assert e.value.status == 8
        filler.clear()
        torch.cuda.empty_cache()
        rsv.rsv_set_frequencies(op, w.omegas)
        rsv.rsv_march_direct(op, x, w.k, z, **rsv.march_opts_for(w))
        assert torch.equal(y, z)
    finally:
        filler.clear()
        torch.cuda.empty_cache()
        rsv.rsv_destroy_operator(op)
