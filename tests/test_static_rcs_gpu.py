"""The allocation-free PCG on reduced camera systems as an adjustment forms them
(lambda = 1e-4, not diagonally dominant), to the 1e-6 of its callers.

The additions into q come in any order, so the iterates differ between runs and
the stop may fall a few iterations apart: near it the recurrence's residual
moves by a few percent per iteration, up as well as down.  What every run has to
keep, against the Sec. 3.2 recurrence in numpy FP64 on the same system:

* the true residual: the recurrence's is at most tol ||b||, and the two part by
  at most k 2^-24 || |S| |x| || after k FP32 iterations (Greenbaum's bound, the
  iterates' norms growing towards ||x||);
* the iterations: FP32 loses conjugacy, which delays the stop and cannot bring
  it forward by more than the plateaus of the residual near it (a tenth); with
  less than half as many again the FP32 recurrence still follows the FP64 one;
* the status, and the same from a second call on the shared scratch."""
import numpy as np
import pytest

import scenes
from test_pcg_sizes_gpu import pcg, product

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("along,across,seed", [(6, 4, 11), (11, 6, 12), (20, 10, 13)])
def test_static_pcg_on_reduced_camera_systems(along, across, seed):
    import torch

    from paper_2307_08383_gb300.build import build
    build()
    import paper_2307_08383_gb300 as B
    s = scenes.aerial_small(along, across, pts_per_cam=50, seed=seed)
    g = B.Problem(s.cams0, s.pts0, s.obs_cam, s.obs_pt, s.obs_uv, precision=B.BA_FP64)
    g.linearize()
    g.form_rcs(1e-4)
    row_ptr, col, val, b = g.rcs()
    g.close()
    val, b = val.astype(np.float32), b.astype(np.float32)
    S, rhs, n, tol = val.astype(np.float64), b.astype(np.float64), along * across, 1e-6
    _, k64 = pcg(row_ptr, col, S, rhs, tol)
    dev = [torch.from_numpy(a).cuda() for a in (row_ptr, col, val, b)]
    x = torch.empty(n, 6, device="cuda")
    for _ in range(4):
        status, its, rel = B.ba_pcg_solve_static(n, len(col), *[t.data_ptr() for t in dev], x.data_ptr(), tol, 0,
                                                 torch.cuda.current_stream().cuda_stream)
        assert status == B.BA_OK and rel <= tol
        assert 0.9 * k64 - 1 <= its <= 2 * k64, (its, k64)
        y = x.cpu().numpy().astype(np.float64)
        drift = its * 2.0 ** -24 * np.linalg.norm(product(row_ptr, col, np.abs(S), np.abs(y)))
        assert np.linalg.norm(rhs - product(row_ptr, col, S, y)) <= tol * np.linalg.norm(rhs) + drift
