"""FP32 results that have to keep their bits.

An FP32 system's last bits decide where an LM trajectory goes some steps on (and
how many PCG iterations it takes), so a change of the order of addition or of a
rounding in the FP32 path is not a matter of a tolerance.  The digests are
SHA-256 over the FP32 values, recorded with CUDA 13.0 from the kernels that sum
each block's products and partials in list order, damp the diagonal by one fused
multiply-add and cut the split CG's entries into the passes of a grid of CTAs.
Inputs are rounded to short binary fractions, so that they do not depend on the
host's mathematical functions."""
import hashlib

import numpy as np
import pytest

import scenes
from test_pcg_sizes_gpu import banded_pattern
from test_vb_sizes_gpu import sizes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2307_08383_gb300.build import build
    build()
    import paper_2307_08383_gb300 as mod
    return mod


def digest(*arrays):
    h = hashlib.sha256()
    for a in arrays:
        h.update(np.ascontiguousarray(a, dtype=np.float32).tobytes())
    return h.hexdigest()[:16]


def rounded(a, bits):
    return np.round(np.asarray(a) * 2.0 ** bits) / 2.0 ** bits


def adjustment(B, kind, size, seed, **kw):
    s = (scenes.ring_scene(n_cams=size, n_pts=40 * size, seed=seed) if kind == "ring"
         else scenes.aerial_small(size, size // 2, pts_per_cam=60, seed=seed))
    return B.Problem(rounded(s.cams0, 20), rounded(s.pts0, 20), s.obs_cam, s.obs_pt, rounded(s.obs_uv, 10),
                     precision=B.BA_FP32, **kw)


FORMED = {
    ("ring", 8, 1): "f925c2f67da42085",
    ("ring", 40, 2): "e6bac43c56223308",
    ("aerial", 8, 3): "0ed7784669abbf97",
    ("aerial", 24, 4): "6536b2073cab8830"}


def formed(B, kind, size, seed):
    g = adjustment(B, kind, size, seed)
    g.linearize()
    g.form_rcs(1e-4)
    _, _, val, b = g.rcs()
    g.close()
    return digest(val, b)


@pytest.mark.parametrize("kind,size,seed", list(FORMED))
def test_formed_system(B, kind, size, seed):
    assert formed(B, kind, size, seed) == FORMED[kind, size, seed]


SOLVED = {
    (1, 1): "6b60bac415ca7841",
    (2, 1): "81bce8132a56b548",
    (24, 23): "9b64ab87d92c6a6b",
    (60, 59): "0f582ece9e37bb23",
    (128, 58): "c9216e937f2322e1",
    (160, 75): "f11d1d32d91d7a0f",
    (200, 33): "e2d9e2800fe43be4",
    (1300, 5): "890af9b61d8e3c73",
    (1700, 5): "86c8c95352b3c85e",
    (2400, 2): "adba1a73e1fa99a8",
    (4000, 2): "cf6f9ce1e7e9fff3"}


def integer_system(row_ptr, col, cdim, seed):
    """Values and right-hand side of few bits: off-diagonal entries k / 16, |k| <= 8,
    diagonal blocks symmetric with a diagonal above the sums of their rows."""
    rng = np.random.default_rng(seed)
    row = np.repeat(np.arange(len(cdim)), np.diff(row_ptr))
    blocks, total = [], np.zeros(len(cdim), np.int64)
    for i, j in zip(row, col):
        k = rng.integers(-8, 9, (cdim[i], cdim[j]))
        blocks.append(np.tril(k) + np.tril(k, -1).T if i == j else k)
        total[i] += np.abs(k).sum(1).max()
        if i != j:
            total[j] += np.abs(k).sum(0).max()
    for i in range(len(cdim)):
        k = row_ptr[i]
        d = blocks[k] - np.diag(np.diag(blocks[k]))
        blocks[k] = d + np.diag(total[i] + np.abs(d).sum(1) + rng.integers(1, 40, cdim[i]))
    val = np.concatenate([k.reshape(-1) for k in blocks]) / 16.0
    return val, rng.integers(-200, 201, int(np.sum(cdim))) / 16.0


def solved(B, n, half):
    row_ptr, col = banded_pattern(n, half)
    val, b = integer_system(row_ptr, col, np.full(n, 6, np.int32), 9600 + n)
    g = B.Problem.from_rcs(row_ptr, col, val.reshape(-1, 6, 6), b.reshape(n, 6), precision=B.BA_FP32, pcg_rel_tol=1e-6)
    out = [g.solve_rcs()[0]["pcg_iters"], g.step()[0]]
    g.close()
    return digest(*out)


@pytest.mark.parametrize("n,half", list(SOLVED))
def test_solved_system(B, n, half):
    assert solved(B, n, half) == SOLVED[n, half]


STEPPED = {
    ("ring", 8, 1, 1e-2): "0565fe2ffdcc72e1",
    ("ring", 16, 2, 1e-2): "5f09f9b988710b05",
    ("ring", 40, 5, 1e-2): "0feb3c9e1128c962",
    ("aerial", 8, 3, 0.1): "35d00e0f43339726",
    ("aerial", 12, 6, 0.1): "328506db7bfe5236",
    ("aerial", 20, 7, 0.1): "61170a5853468066",
    ("aerial", 30, 8, 0.1): "d23b1b022fb034cf"}


def stepped(B, kind, size, seed, tol):
    g = adjustment(B, kind, size, seed, pcg_rel_tol=tol)
    out = []
    for _ in range(3):
        info = g.lm_step()
        out += [info["pcg_iters"], info["accepted"], info["cost_after"], *g.step()]
    g.close()
    return digest(*out)


@pytest.mark.parametrize("kind,size,seed,tol", list(STEPPED))
def test_lm_steps(B, kind, size, seed, tol):
    assert stepped(B, kind, size, seed, tol) == STEPPED[kind, size, seed, tol]


VARIABLE = {
    (40, 30, "any"): "3bab62ea3c32c13e",
    (90, 12, "6"): "c089feef167bdc76",
    (330, 9, "mixed"): "00b12007f81d0148",
    (700, 22, "mixed"): "a964c4219b711fb8",
    (400, 5, "any"): "5b93de694b78c5ed",
    (60, 20, "16"): "7435aab8a39ddd9d",
    (3000, 4, "1"): "aadc50e04a404946",
    (5200, 1, "any"): "d6fd02df987c0560"}


def variable(B, n, half, kind):
    row_ptr, col = banded_pattern(n, half)
    cdim = sizes(kind, n, 77 + n)
    val, b = integer_system(row_ptr, col, cdim, 9700 + n)
    g = B.VBSMC(cdim, row_ptr, col, val, b, precision=B.BA_FP32)
    x, its = g.solve(1e-5)[:2]
    g.close()
    return digest(its, x)


@pytest.mark.parametrize("n,half,kind", list(VARIABLE))
def test_variable_size_system(B, n, half, kind):
    assert variable(B, n, half, kind) == VARIABLE[n, half, kind]


INTERIORS = {
    (5, 4, 0.5, 1): "cd94822313b22174",
    (8, 5, 0.1, 2): "7a12002e595f49d3",
    (12, 6, 1.0, 3): "63c87248ade01d32"}


def interiors(B, along, across, frac, seed):
    s = scenes.aerial_small(along, across, pts_per_cam=60, seed=9800 + seed)
    intr = rounded(scenes.interiors0(s.n_cams, seed=seed), 20)
    g = B.VBIProblem(rounded(s.cams0, 20), intr, scenes.block_sizes(s.n_cams, frac, seed), rounded(s.pts0, 20), s.obs_cam,
                     s.obs_pt, rounded(s.obs_uv, 10), precision=B.BA_FP32, pcg_rel_tol=0.1)
    out = []
    for _ in range(2):
        info = g.lm_step()
        out += [info["pcg_iters"], info["accepted"], info["cost_after"], *g.step()]
    g.close()
    return digest(*out)


@pytest.mark.parametrize("along,across,frac,seed", list(INTERIORS))
def test_lm_steps_with_interiors(B, along, across, frac, seed):
    assert interiors(B, along, across, frac, seed) == INTERIORS[along, across, frac, seed]
