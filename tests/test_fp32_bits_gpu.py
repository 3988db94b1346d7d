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
