"""Block-Jacobi PCG over the launch shapes its kernels choose by size.

A given system (``Problem.from_rcs``) with seeded SPD values, at camera counts
on both sides of the lines where the kernels change the warps per CTA, the
warps per row or the grid.  The reference is the recurrence of Sec. 3.2 in
numpy FP64.  Tolerances: the solve stops at ||r|| <= 1e-10 ||b|| by its own
recurrence, whose residual and the true one differ by rounding of the iterates
(n_iter * 2^-53 * cond, below 1e-13 for these diagonally dominant systems), so
||b - S x|| <= 1.01e-10 ||b||; iteration counts agree within one; two iterates
with residuals of 1e-10 differ by at most 2e-10 cond(S), and block dominance
bounds cond(S) by the ratio of the largest to the smallest diagonal block
eigenvalue times (1 + s) / (1 - s), s < 1 / 2 the share of a row's norm sum in
its diagonal: 1e-8 covers the ratios these seeds have (below 50)."""
import numpy as np
import pytest

import scenes

pytestmark = pytest.mark.gpu


def banded_pattern(n, half):
    """Every row coupled to four fifths of the next ``half`` cameras."""
    row_ptr, col = [0], []
    for i in range(n):
        c = [i] + [j for j in range(i + 1, min(n, i + half + 1)) if (i * 7 + j) % 5]
        col += c
        row_ptr.append(len(col))
    return np.array(row_ptr, np.int32), np.array(col, np.int32)


def system(n, half, seed):
    row_ptr, col = banded_pattern(n, half)
    val, _ = scenes.random_block_spd(row_ptr, col, np.full(n, 6, np.int32), seed)
    b = np.random.default_rng(seed + 1).standard_normal((n, 6))
    return row_ptr, col, val.reshape(-1, 6, 6), b


def product(row_ptr, col, val, x):
    row = np.repeat(np.arange(len(row_ptr) - 1), np.diff(row_ptr))
    y = np.zeros_like(x)
    np.add.at(y, row, np.einsum("kab,kb->ka", val, x[col]))
    off = row != col
    np.add.at(y, col[off], np.einsum("kba,kb->ka", val[off], x[row[off]]))
    return y


def pcg(row_ptr, col, val, b, tol):
    Minv = np.linalg.inv(val[row_ptr[:-1]])
    x, r = np.zeros_like(b), b.copy()
    z = np.einsum("nab,nb->na", Minv, r)
    d, rz, r0 = z, float((r * z).sum()), np.linalg.norm(b)
    for it in range(1, 10000):
        q = product(row_ptr, col, val, d)
        a = rz / float((d * q).sum())
        x, r = x + a * d, r - a * q
        if np.linalg.norm(r) <= tol * r0:
            return x, it
        z = np.einsum("nab,nb->na", Minv, r)
        new = float((r * z).sum())
        d, rz = z + new / rz * d, new
    raise AssertionError("no convergence")


@pytest.mark.parametrize("n,half", [(1, 1), (2, 1), (3, 2), (40, 39), (152, 9), (153, 20), (305, 45), (609, 12),
                                    (1217, 6), (2500, 4), (130, 129)])
def test_fp64_pcg_over_launch_shapes(n, half):
    from paper_2307_08383_gb300.build import build
    build()
    import paper_2307_08383_gb300 as B
    row_ptr, col, val, b = system(n, half, 9100 + n)
    tol = 1e-10
    ref, its = pcg(row_ptr, col, val, b, tol)
    g = B.Problem.from_rcs(row_ptr, col, val, b, precision=B.BA_FP64, pcg_rel_tol=tol)
    for _ in range(2):  # a second solve finds nothing of the first
        info, conv = g.solve_rcs()
        assert conv and abs(info["pcg_iters"] - its) <= 1, (info["pcg_iters"], its)
        x = g.step()[0].reshape(n, 6)
        assert np.linalg.norm(b - product(row_ptr, col, val, x)) <= 1.01 * tol * np.linalg.norm(b)
        assert np.linalg.norm(x - ref) <= 1e-8 * np.linalg.norm(ref)
    g.close()


@pytest.mark.parametrize("n,half,shift", [(1, 1, 0), (7, 6, 1), (153, 20, 0), (200, 199, 0), (200, 199, 1),
                                          (1300, 33, 0), (8192, 3, 1)])
def test_static_pcg_over_launch_shapes(n, half, shift):
    """The allocation-free solve: one to 54 rows per CTA, rows of more than a
    warp's blocks, CTAs whose blocks exceed their shared memory share, and
    arrays at a 4-byte offset (shift).  FP32 recurrence to 1e-5: the true
    residual is within 100 eps of it."""
    import torch

    from paper_2307_08383_gb300.build import build
    build()
    import paper_2307_08383_gb300 as B
    row_ptr, col, val, b = system(n, half, 9200 + n)
    val, b = val.astype(np.float32), b.astype(np.float32)
    dev = [torch.from_numpy(row_ptr).cuda(), torch.from_numpy(col).cuda()]
    flat = [torch.zeros(a.size + 1, device="cuda") for a in (val, b, b)]
    for t, a in zip(flat[:2], (val, b)):
        t[shift:shift + a.size] = torch.from_numpy(a.reshape(-1)).cuda()
    ptr = [t.data_ptr() + 4 * shift for t in flat]
    for _ in range(2):
        status, its, rel = B.ba_pcg_solve_static(n, len(col), dev[0].data_ptr(), dev[1].data_ptr(), ptr[0], ptr[1],
                                                 ptr[2], 1e-5, 0, torch.cuda.current_stream().cuda_stream)
        assert status == B.BA_OK and 1 <= its < 40 and rel <= 1e-5
        x = flat[2][shift:shift + b.size].cpu().numpy().astype(np.float64).reshape(n, 6)
        r = b - product(row_ptr, col, val.astype(np.float64), x)
        assert np.linalg.norm(r) <= (1e-5 + 100 * np.finfo(np.float32).eps) * np.linalg.norm(b)


@pytest.mark.parametrize("n,half", [(3, 2), (152, 9), (200, 199)])
def test_fp64_pcg_without_mailboxes(n, half):
    """A cap on device memory that the mailboxes would exceed: the loop that
    exchanges by counters solves the same systems."""
    from paper_2307_08383_gb300.build import build
    build()
    import paper_2307_08383_gb300 as B
    row_ptr, col, val, b = system(n, half, 9100 + n)
    ref, its = pcg(row_ptr, col, val, b, 1e-10)
    g = B.Problem.from_rcs(row_ptr, col, val, b, precision=B.BA_FP64, pcg_rel_tol=1e-10, device_mem_cap=1)
    info, conv = g.solve_rcs()
    assert conv and abs(info["pcg_iters"] - its) <= 1
    assert np.linalg.norm(g.step()[0].reshape(n, 6) - ref) <= 1e-8 * np.linalg.norm(ref)
    g.close()


@pytest.mark.parametrize("n,half", [(1, 1), (2, 1), (24, 23), (128, 60), (160, 63), (160, 75), (1500, 20),
                                    (2600, 40), (2600, 62)])
def test_fp32_split_cg_over_launch_shapes(n, half):
    """FP32: one cluster (up to 14,336 off-diagonal entries) and a CTA per SM;
    passes held in shared memory and passes copied again each iteration.  The
    refinement stops at a true residual of 1e-6 ||b||; the step is returned
    in FP32, which adds at most 2^-24 ||S|| ||x|| <= 2^-24 cond(S) ||b||,
    cond(S) < 150 (see above)."""
    from paper_2307_08383_gb300.build import build
    build()
    import paper_2307_08383_gb300 as B
    row_ptr, col, val, b = system(n, half, 9300 + n)
    val, b = val.astype(np.float32).astype(np.float64), b.astype(np.float32).astype(np.float64)
    g = B.Problem.from_rcs(row_ptr, col, val, b, precision=B.BA_FP32, pcg_rel_tol=1e-6)
    for _ in range(2):
        info, conv = g.solve_rcs()
        assert conv and 1 <= info["pcg_iters"] < 200
        x = g.step()[0].reshape(n, 6)
        assert np.linalg.norm(b - product(row_ptr, col, val, x)) <= (1e-6 + 150 * 2.0 ** -24) * np.linalg.norm(b)
    g.close()


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("cams,pts", [(8, 60), (16, 2500), (40, 6000)])
def test_group_sizes_from_the_problem(prec, cams, pts):
    """Point groups sized by the problem against the largest ones: the same
    system, its sums in another order (64 cameras' worth of terms a block at
    most 2^13 eps of the block's norm)."""
    from paper_2307_08383_gb300.build import build
    build()
    import paper_2307_08383_gb300 as B
    s = scenes.ring_scene(n_cams=cams, n_pts=pts, seed=9400 + cams)
    out = []
    for kw in ({}, {"group_max_obs": 512}):
        g = B.Problem(s.cams0, s.pts0, s.obs_cam, s.obs_pt, s.obs_uv,
                      precision=B.BA_FP64 if prec == "fp64" else B.BA_FP32, **kw)
        g.linearize()
        g.form_rcs(1e-4)
        out.append((g.stats()["n_groups"], *g.rcs()))
        g.close()
    assert out[0][0] >= out[1][0]
    eps = np.finfo(np.float64 if prec == "fp64" else np.float32).eps
    for a, c in zip(out[0][3:], out[1][3:]):
        assert np.abs(np.asarray(a) - np.asarray(c)).max() <= 2 ** 13 * eps * np.abs(np.asarray(c)).max()
