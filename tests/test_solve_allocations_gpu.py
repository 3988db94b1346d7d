"""An FP64 solve by the Sec. 3.2 recurrence allocates nothing, its first run
included: ba_stats.device_bytes, which every allocation of a problem adds to, is
the same before and after, for the loop in registers, the loop with counters and
rows that no register loop takes."""
import pytest

from test_pcg_sizes_gpu import system

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,half,kw", [(40, 39, {}), (40, 39, {"device_mem_cap": 1}), (305, 200, {}), (1217, 6, {})])
def test_first_fp64_solve_allocates_nothing(n, half, kw):
    from paper_2307_08383_gb300.build import build
    build()
    import paper_2307_08383_gb300 as B
    row_ptr, col, val, b = system(n, half, 9800 + n)
    g = B.Problem.from_rcs(row_ptr, col, val, b, precision=B.BA_FP64, pcg_rel_tol=1e-10, **kw)
    before = g.stats()["device_bytes"]
    for _ in range(2):
        assert g.solve_rcs()[1]
        assert g.stats()["device_bytes"] == before
    g.close()
