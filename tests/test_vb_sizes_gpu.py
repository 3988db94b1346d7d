"""Variable-size BSMC product, M^-1 and PCG over the launch shapes and block
sizes its kernels distinguish: 1 to 16 unknowns per camera in one system, one
to many block rows per CTA, values in shared memory or not, and CTAs that own
more vector entries than threads.  Reference: numpy FP64 on the blocks padded
to 16 x 16.  Tolerances: a product sums at most 32 x 16 terms, so it is within
512 eps of sum |S| |x| per entry; the solves stop at ||r|| <= tol ||b|| by
their own recurrence, and for these block-dominant systems (condition below
50, a few tens of iterations) the true residual is within 100 eps of it
relative to ||b|| in the storage precision."""
import numpy as np
import pytest

import scenes
from test_pcg_sizes_gpu import banded_pattern

pytestmark = pytest.mark.gpu


def padded(row_ptr, col, cdim, val):
    row = np.repeat(np.arange(len(cdim)), np.diff(row_ptr))
    S = np.zeros((len(col), 16, 16))
    size = cdim[row].astype(np.int64) * cdim[col]
    at = np.concatenate([[0], np.cumsum(size)])
    for k in range(len(col)):
        S[k, :cdim[row[k]], :cdim[col[k]]] = val[at[k]:at[k + 1]].reshape(cdim[row[k]], cdim[col[k]])
    return row, S


def product(row, col, S, x):
    y = np.zeros_like(x)
    np.add.at(y, row, np.einsum("kab,kb->ka", S, x[col]))
    off = row != col
    np.add.at(y, col[off], np.einsum("kba,kb->ka", S[off], x[row[off]]))
    return y


def sizes(kind, n, seed):
    rng = np.random.default_rng(seed)
    if kind == "any":
        return rng.integers(1, 17, n).astype(np.int32)
    if kind == "mixed":
        return np.where(rng.random(n) < 0.5, 11, 6).astype(np.int32)
    return np.full(n, int(kind), np.int32)


@pytest.mark.parametrize("n,half,kind,fp32", [(1, 1, "any", False), (3, 2, "any", False), (40, 30, "any", False),
                                              (40, 30, "any", True), (153, 11, "mixed", False),
                                              (400, 25, "11", False), (1000, 9, "mixed", True),
                                              (1600, 22, "11", True), (5200, 1, "16", False), (5200, 1, "16", True),
                                              (330, 3, "1", True), (17, 16, "5", False)])
def test_vb_system_over_sizes(n, half, kind, fp32):
    import torch

    from paper_2307_08383_gb300.build import build
    build()
    import paper_2307_08383_gb300 as B
    row_ptr, col = banded_pattern(n, half)
    cdim = sizes(kind, n, 77 + n)
    T = np.float32 if fp32 else np.float64
    val, _ = scenes.random_block_spd(row_ptr, col, cdim, 9300 + n)
    val = val.astype(T).astype(np.float64)
    N = int(cdim.sum())
    rng = np.random.default_rng(n)
    b = rng.standard_normal(N).astype(T).astype(np.float64)
    x = rng.standard_normal(N).astype(T).astype(np.float64)
    live = np.arange(16)[None] < cdim[:, None]
    row, S = padded(row_ptr, col, cdim, val)

    def pad(v):
        p = np.zeros((n, 16))
        p[live] = v
        return p

    eps = np.finfo(T).eps
    g = B.VBSMC(cdim, row_ptr, col, val, b, precision=B.BA_FP32 if fp32 else B.BA_FP64)
    dx = torch.from_numpy(x.astype(T)).cuda()
    dy = torch.full_like(dx, float("nan"))
    g.spmv(dx, dy)
    y = dy.cpu().numpy().astype(np.float64)
    bound = product(row, col, np.abs(S), pad(np.abs(x)))[live]
    assert np.all(np.abs(y - product(row, col, S, pad(x))[live]) <= 512 * eps * bound)
    tol = 1e-5 if fp32 else 1e-11
    for _ in range(2):  # a second solve finds nothing of the first
        sol, its, rel, _, status = g.solve(tol)
        assert status == B.BA_OK and 1 <= its < 100 and rel <= tol
        r = pad(b) - product(row, col, S, pad(sol))
        assert np.linalg.norm(r) <= (tol + 100 * eps) * np.linalg.norm(b)
    # a diagonal block that is not positive definite is still refused
    bad = val.copy()
    k = int(row_ptr[n - 1])
    at = np.concatenate([[0], np.cumsum(cdim[row].astype(np.int64) * cdim[col])])
    c = int(cdim[n - 1])
    bad[at[k] + c * c - 1] = -1.0
    with pytest.raises(B.BAError) as ei:
        B.VBSMC(cdim, row_ptr, col, bad, b, precision=B.BA_FP32 if fp32 else B.BA_FP64)
    assert ei.value.status == B.BA_ERR_NOT_SPD
    g.close()


def test_interiors_state_round_trip():
    """The state set and read back bit for bit, unchanged by a refused one, and
    the LM step from it the same."""
    from paper_2307_08383_gb300.build import build
    build()
    import paper_2307_08383_gb300 as B
    s = scenes.shuffled(scenes.aerial_small(n_along=5, n_across=4, pts_per_cam=30, seed=9500), 3)
    intr = scenes.interiors0(s.n_cams, seed=9501)
    args = (s.cams0, intr, np.full(s.n_cams, 11, np.int32), s.pts0, s.obs_cam, s.obs_pt, s.obs_uv)
    ref = B.VBIProblem(*args, precision=B.BA_FP64)
    g = B.VBIProblem(*args, precision=B.BA_FP64)
    want = ref.lm_step()
    rng = np.random.default_rng(9502)
    cams, ins, pts = (a + 1e-3 * rng.standard_normal(a.shape) for a in (s.cams0, intr, s.pts0))
    g.set_state(cams, ins, pts, 1e-3, 2.0)
    for a, b in zip(g.state(), (cams, ins, pts)):
        assert np.array_equal(a.reshape(b.shape), b)
    for k, v in ((0, np.nan), (pts.size - 1, np.inf)):
        bad = pts.copy()
        bad.flat[k] = v
        with pytest.raises(B.BAError):
            g.set_state(s.cams0, intr, bad, 1e-3, 2.0)
        for a, b in zip(g.state(), (cams, ins, pts)):
            assert np.array_equal(a.reshape(b.shape), b)
    g.set_state(s.cams0, intr, s.pts0, 1e-4, 2.0)
    info = g.lm_step()
    assert (info["cost_before"], info["accepted"]) == (want["cost_before"], want["accepted"])
    assert abs(info["cost_after"] - want["cost_after"]) <= 1e-12 * want["cost_after"]
    for a, b in zip(g.step(), ref.step()):
        assert np.linalg.norm(a - b) <= 1e-9 * np.linalg.norm(b)
    ref.close()
    g.close()
