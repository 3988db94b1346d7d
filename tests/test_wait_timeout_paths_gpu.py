"""The bounded waits of the PCG launch shapes that test_wait_timeout_gpu does not
reach: its 16 cameras solve in one thread-block cluster (FP32 split; an mbarrier
that expects one arrival too many) and in the register-resident loop (FP64;
mailboxes read for a tag that nobody posts).  Here the split CG on the grid
(more than 14,336 off-diagonal entries) and the FP64 loop whose CTAs exchange by
arrival counters (a cap that leaves no room for mailboxes; rows too long for a
CTA's registers), both with the counters one arrival short.  Every wait ends by
its own limit, about a millisecond."""
import numpy as np
import pytest

from test_pcg_sizes_gpu import system

pytestmark = pytest.mark.gpu

LIMIT = 2_000_000  # SM cycles


@pytest.mark.parametrize("prec,n,half,kw", [("fp32", 200, 199, {}), ("fp32", 2600, 40, {}),
                                            ("fp64", 16, 15, {"device_mem_cap": 1}), ("fp64", 305, 200, {}),
                                            ("fp64", 1217, 6, {})])
def test_wait_runs_out(prec, n, half, kw):
    import torch

    from paper_2307_08383_gb300.build import build
    build()
    import paper_2307_08383_gb300 as B
    row_ptr, col, val, b = system(n, half, 9700 + n)
    if prec == "fp32":
        off = 2 * (len(col) - n)
        assert off > 14336
        val, b = val.astype(np.float32).astype(np.float64), b.astype(np.float32).astype(np.float64)

    def problem():
        return B.Problem.from_rcs(row_ptr, col, val, b, precision=B.BA_FP32 if prec == "fp32" else B.BA_FP64,
                                  pcg_rel_tol=1e-6, **kw)

    ref = problem()
    assert ref.solve_rcs()[1]
    want = ref.step()[0]
    ref.close()
    g = problem()
    g.arm_wait_timeout(LIMIT)
    with pytest.raises(B.BAError) as ei:
        g.solve_rcs()
    assert ei.value.status == B.BA_ERR_TIMEOUT
    with pytest.raises(B.BAError) as ei:
        g.solve_rcs()
    assert ei.value.status == B.BA_ERR_STATE
    g.close()
    torch.cuda.synchronize()  # the context answers: no kernel is left waiting
    h = problem()
    assert h.solve_rcs()[1]
    assert np.array_equal(h.step()[0], want)
    h.close()
