"""Point groups of other sizes than the default.

FP32 with small groups given: the sums of a block over more partials, each in
another order than with the largest groups, agree within 2^13 eps of the
block's norm (at most 40 cameras' observations, a few thousand terms a block).

FP64 under a cap on device memory: the groups that are sized for the device's
SMs write more partials than the largest ones; a cap that only they exceed gets
the largest, and then S and b are those of that group size bit for bit; a cap
below that is refused."""
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


def formed(B, s, **kw):
    g = B.Problem(s.cams0, s.pts0, s.obs_cam, s.obs_pt, s.obs_uv, **kw)
    g.linearize()
    g.form_rcs(1e-4)
    out = (g.stats(), *g.rcs())
    g.close()
    return out


@pytest.mark.parametrize("cams,pts,size", [(8, 60, 32), (16, 2500, 64), (40, 6000, 104)])
def test_fp32_small_groups(B, cams, pts, size):
    s = scenes.ring_scene(n_cams=cams, n_pts=pts, seed=9400 + cams)
    small = formed(B, s, precision=B.BA_FP32, group_max_obs=size)
    large = formed(B, s, precision=B.BA_FP32, group_max_obs=512)
    assert small[0]["n_groups"] > large[0]["n_groups"]
    for a, c in zip(small[3:], large[3:]):
        assert np.abs(a - c).max() <= 2 ** 13 * np.finfo(np.float32).eps * np.abs(c).max()


def test_fp64_groups_under_a_memory_cap(B):
    s = scenes.ring_scene(n_cams=40, n_pts=6000, seed=9440)
    own = formed(B, s, precision=B.BA_FP64)
    large = formed(B, s, precision=B.BA_FP64, group_max_obs=512)
    assert own[0]["n_groups"] > large[0]["n_groups"]
    seen = []
    for cap in np.linspace(0.9 * large[0]["device_bytes"], 1.1 * own[0]["device_bytes"], 24).astype(int):
        try:
            got = formed(B, s, precision=B.BA_FP64, device_mem_cap=int(cap))
        except B.BAError as e:
            assert e.status == B.BA_ERR_OOM
            seen.append(0)
            continue
        assert got[0]["device_bytes"] <= cap * (1 + 1e-3)
        ref = own if got[0]["n_groups"] == own[0]["n_groups"] else large
        assert got[0]["n_groups"] == ref[0]["n_groups"] and got[0]["n_partials"] == ref[0]["n_partials"]
        for a, c in zip(got[1:], ref[1:]):
            assert np.array_equal(a, c)
        seen.append(2 if ref is own else 1)
    assert seen == sorted(seen) and set(seen) == {0, 1, 2}
