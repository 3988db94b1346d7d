"""Measured workloads of the bundle-adjustment library, through its Python binding.

Each case is a call, or a short run of calls, that a user of the library makes:

* ``lm``        LM iterations of an adjustment with six unknowns per camera: the
                state in (``set_state``), some ``lm_step``, the state out;
* ``interiors`` the same with interior parameters (``VBIProblem``);
* ``form``      the stages up to the reduced camera system, for a caller with a
                solver of its own: linearize, form the RCS, its product with a
                given vector;
* ``solve``     a given reduced camera system solved (``Problem.from_rcs``);
* ``static``    the same through the allocation-free entry point, all arrays
                the caller's own device buffers;
* ``vbsmc``     a variable-size block system: one product and one solve.

Scenes are those of the repository's generators (cameras on a ring, nadir
grids), made here on the GPU from the seed.  Results of FP64 problems are
returned as they come (FP64); those of FP32 problems, whose Jacobians, systems
and steps are FP32, are returned in FP32.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2307_08383_gb300 as B

F, C = 1000.0, 500.0  # pinhole of every scene: focal length, principal point (px)
DEV = "cuda"
F64 = torch.float64


def listed():
    return [
        # the smallest adjustment: the library's default options (FP64, PCG to
        # 1e-10) on the ring scene of the parity tests; launches and latency
        {"name": "lm_ring50_fp64", "kind": "lm", "scene": "ring", "n": 50, "pts": 2000, "fp32": False,
         "tol": 1e-10, "huber": False, "steps": 1},
        # one flight of images in the default precision
        {"name": "lm_aerial200_fp64", "kind": "lm", "scene": "aerial", "n": 200, "along": 20, "pts": 40000, "fp32": False,
         "tol": 1e-10, "huber": False, "steps": 1},
        # the same flight in FP32, solved to the paper's tolerance: the first three
        # iterations of an adjustment
        {"name": "lm_aerial200_fp32", "kind": "lm", "scene": "aerial", "n": 200, "along": 20, "pts": 40000, "fp32": True,
         "tol": 0.1, "huber": False, "steps": 3},
        # the benchmark's workload: 5,000 cameras, 1M points, about 4.9M observations
        {"name": "lm_aerial5000_fp32", "kind": "lm", "scene": "aerial", "n": 5000, "along": 100, "pts": 1000000, "fp32": True,
         "tol": 0.1, "huber": False, "steps": 3},
        # formation of the RCS alone at an uneven middle size, and in FP64 with the
        # robust loss and 1 % outliers
        {"name": "form_aerial1770_fp32", "kind": "form", "scene": "aerial", "n": 1770, "along": 59, "pts": 355000, "fp32": True,
         "huber": False},
        {"name": "form_aerial450_fp64", "kind": "form", "scene": "aerial", "n": 450, "along": 30, "pts": 45000, "fp32": False,
         "huber": True},
        # solves of a given system, FP32 sweeps refined to the tolerance of the
        # smoke check: a small one, and one of the size of the solver benchmark's
        # held-out systems
        {"name": "solve_128_fp32", "kind": "solve", "n": 128, "along": 16, "pts": 12800, "tol": 1e-12},
        {"name": "solve_2556_fp32", "kind": "solve", "n": 2556, "along": 71, "pts": 127800, "tol": 1e-12},
        # the allocation-free solver, to the tolerance its tests use
        {"name": "static_1250", "kind": "static", "n": 1250, "along": 50, "pts": 62500, "tol": 1e-6},
        # self-calibration: five interiors per camera on every camera (FP32, as
        # the benchmark runs it; started with more damping than the poses alone,
        # since focal lengths and heights trade off), and on half of them (FP64)
        {"name": "interiors990_fp32", "kind": "interiors", "n": 990, "along": 45, "pts": 99000, "fp32": True, "frac": 1.0,
         "tol": 0.1, "lam": 1e-2, "steps": 2},
        {"name": "interiors120_fp64", "kind": "interiors", "n": 120, "along": 15, "pts": 12000, "fp32": False, "frac": 0.5,
         "tol": 1e-10, "lam": 1e-4, "steps": 1},
        # the benchmark's variable-size system at c = 11, with fewer cameras
        {"name": "vbsmc1984_fp32", "kind": "vbsmc", "n": 1984, "along": 62, "fp32": True, "frac": 1.0, "tol": 1e-6},
    ]


def _grid(rng, lo, hi):
    """A flight grid of about lo .. hi cameras, half as many across as along."""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    across = max(2, int(round(math.sqrt(n / 2))))
    along = max(2, int(n / across))
    return {"n": across * along, "along": along}


def draw(rng):
    kind = rng.choice(["lm", "lm", "form", "solve", "static", "interiors", "vbsmc"])
    fp32 = rng.random() < 0.6
    if kind == "lm" and rng.random() < 0.25:
        n = int(round(math.exp(rng.uniform(math.log(8), math.log(120)))))
        return {"kind": kind, "scene": "ring", "n": n, "pts": n * rng.randint(25, 60), "fp32": fp32,
                "tol": 1e-2 if fp32 else 1e-10, "huber": False, "steps": 1}
    if kind == "lm":
        g, huber = _grid(rng, 30, 4000 if fp32 else 400), rng.random() < 0.5
        return {"kind": kind, "scene": "aerial", **g, "pts": g["n"] * rng.randint(50, 200), "fp32": fp32,
                "tol": 0.1 if fp32 else 1e-10, "huber": huber,
                "steps": rng.randint(1, 3) if fp32 and not huber else 1}
    if kind == "form":
        g = _grid(rng, 30, 4000 if fp32 else 800)
        return {"kind": kind, "scene": "aerial", **g, "pts": g["n"] * rng.randint(50, 200), "fp32": fp32,
                "huber": rng.random() < 0.5}
    if kind in ("solve", "static"):
        g = _grid(rng, 24, 4000)
        return {"kind": kind, **g, "pts": 50 * g["n"], "tol": 1e-12 if kind == "solve" else 1e-6}
    if kind == "interiors":
        g = _grid(rng, 30, 1000 if fp32 else 200)
        return {"kind": kind, **g, "pts": g["n"] * rng.randint(50, 100), "fp32": fp32,
                "frac": rng.choice([1.0, 0.5, 0.1]), "tol": 0.1 if fp32 else 1e-10,
                "lam": 1e-2 if fp32 else 1e-4, "steps": rng.randint(1, 2) if fp32 else 1}
    return {"kind": kind, **_grid(rng, 50, 2500), "fp32": fp32, "frac": rng.choice([1.0, 0.5]),
            "tol": 1e-6 if fp32 else 1e-12}


# ---------------------------------------------------------------------------
# scenes: cameras [omega, t] with X_cam = R(omega) X + t, points, observations
# ---------------------------------------------------------------------------

def _qmul(a, b):
    w, x, y, z = a.unbind(-1)
    W, X, Y, Z = b.unbind(-1)
    return torch.stack([w * W - x * X - y * Y - z * Z, w * X + x * W + y * Z - z * Y,
                        w * Y - x * Z + y * W + z * X, w * Z + x * Y - y * X + z * W], -1)


def _qexp(v):
    th = v.norm(dim=-1, keepdim=True)
    return torch.cat([torch.cos(th / 2), 0.5 * v * torch.sinc(th / (2 * math.pi))], -1)


def _qlog(q):
    q = torch.where(q[..., :1] < 0, -q, q)
    s = q[..., 1:].norm(dim=-1, keepdim=True)
    f = torch.where(s < 1e-12, 2.0 / q[..., :1], 2.0 * torch.atan2(s, q[..., :1]) / s.clamp_min(1e-300))
    return f * q[..., 1:]


def _qrot(q):
    w, x, y, z = q.unbind(-1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], -1).view(*q.shape[:-1], 3, 3)


def _tracks(g, P, cap):
    """Track lengths 2 + Geometric with mean 5, at most 20 and cap."""
    u = torch.rand(P, generator=g, device=DEV, dtype=F64)
    extra = torch.floor(torch.log1p(-u) / math.log(0.75)).to(torch.int64)
    return 2 + torch.where(extra > 18, extra % 19, extra).clamp_max(max(0, min(20, cap) - 2))


def _scene(case, seed):
    """A scene on the GPU: ground truth projected with N(0, 1) px noise (ring:
    0.5 px), and perturbed initial values (0.01 rad, 0.05 m, points 0.1 m)."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed * 7919 + 17)

    def rand(*s):
        return torch.rand(*s, generator=g, device=DEV, dtype=F64)

    def randn(*s):
        return torch.randn(*s, generator=g, device=DEV, dtype=F64)

    n, P = case["n"], case["pts"]
    if case.get("scene") == "ring":
        phi = 2 * math.pi * torch.arange(n, device=DEV, dtype=F64) / n
        ctr = torch.stack([30 * phi.cos(), 30 * phi.sin(), 0 * phi], 1)
        # looking at the centre from phi = 0, turned about the vertical axis by phi
        q0 = torch.tensor([0.5, 0.5, 0.5, -0.5], device=DEV, dtype=F64).expand(n, 4)
        q = _qmul(q0, torch.stack([(phi / 2).cos(), 0 * phi, 0 * phi, -(phi / 2).sin()], 1))
        pts = 10 * rand(P, 3) - 5
        L = 3 + (6 * rand(P)).to(torch.int64).clamp_max(min(5, n - 3))
        near = rand(P, n).topk(min(8, n), dim=1).indices
        noise = 0.5
    else:
        nl, na = case["along"], n // case["along"]
        ix, iy = torch.arange(n, device=DEV) % nl, torch.arange(n, device=DEV) // nl
        ctr = torch.stack([40.0 * ix, 70.0 * iy, torch.full((n,), 100.0, device=DEV)], 1).to(F64)
        yaw = 0.02 * randn(n)
        q = torch.stack([0 * yaw, (yaw / 2).cos(), (yaw / 2).sin(), 0 * yaw], 1)
        x, y = rand(P) * 40.0 * (nl - 1), rand(P) * 70.0 * (na - 1)
        z = 10 * torch.sin(2 * math.pi * x / 500) * torch.sin(2 * math.pi * y / 500)
        pts = torch.stack([x, y, z], 1)
        # the nearest cameras in xy, from a window of the grid around the point
        wl, wa = min(11, nl), min(7, na)
        i0 = (torch.round(x / 40).long() - wl // 2).clamp(0, nl - wl)
        j0 = (torch.round(y / 70).long() - wa // 2).clamp(0, na - wa)
        cap = min(20, wl * wa)
        near = []
        for s in range(0, P, 1 << 18):
            sl = slice(s, min(P, s + (1 << 18)))
            ci = i0[sl, None] + torch.arange(wl, device=DEV)
            cj = j0[sl, None] + torch.arange(wa, device=DEV)
            d2 = ((70.0 * cj[:, :, None] - y[sl, None, None]) ** 2 + (40.0 * ci[:, None, :] - x[sl, None, None]) ** 2)
            ids = (cj[:, :, None] * nl + ci[:, None, :]).flatten(1)
            near.append(ids.gather(1, d2.flatten(1).topk(cap, dim=1, largest=False).indices))
        near = torch.cat(near)
        L = _tracks(g, P, cap)
        noise = 1.0
    keep = torch.arange(near.shape[1], device=DEV) < L[:, None]
    cam = torch.where(keep, near, torch.full_like(near, n)).sort(dim=1).values
    oc = cam[keep]
    op = torch.arange(P, device=DEV)[:, None].expand_as(cam)[keep]
    R = _qrot(q)
    Xc = torch.einsum("mij,mj->mi", R[oc], pts[op] - ctr[oc])
    uv = F * Xc[:, :2] / Xc[:, 2:] + C + noise * randn(len(oc), 2)
    if case.get("huber"):  # 1 % outliers, uniform in the image
        out = rand(len(oc)) < 0.01
        uv = torch.where(out[:, None], 1000 * rand(len(oc), 2), uv)
    q1 = _qmul(_qexp(0.01 * randn(n, 3)), q)
    ctr1 = ctr + 0.05 * randn(n, 3)
    cams = torch.cat([_qlog(q1), -torch.einsum("nij,nj->ni", _qrot(q1), ctr1)], 1)
    intr = None
    if case["kind"] == "interiors":
        intr = torch.stack([F * (1 + 0.01 * randn(n)), C + 2 * randn(n), C + 2 * randn(n), 0.01 * randn(n),
                            0.01 * randn(n)], 1)
        cdim = torch.where(rand(n) < case["frac"], 11, 6).to(torch.int32)
        return {"cams": cams, "pts": pts + 0.1 * randn(len(pts), 3), "oc": oc, "op": op, "uv": uv, "intr": intr,
                "cdim": cdim}
    return {"cams": cams, "pts": pts + 0.1 * randn(len(pts), 3), "oc": oc, "op": op, "uv": uv}


def _host(t, dtype=None):
    a = t.cpu().numpy()
    return a if dtype is None else a.astype(dtype)


def _pinned(t):
    return torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t).numpy()


# ---------------------------------------------------------------------------
# given systems: the RCS of a scene (FP64 sums in a fixed order, rounded to
# FP32, the precision it is solved in), and a seeded variable-size system
# ---------------------------------------------------------------------------

def _segsum(x, key):
    """Sums of the rows of x with equal keys, in stable order: (sums, keys)."""
    order = torch.sort(key, stable=True).indices
    uniq, cnt = torch.unique_consecutive(key[order], return_counts=True)
    return torch.segment_reduce(x[order], "sum", lengths=cnt, axis=0), uniq


def _schur_system(case, seed):
    """BSMC arrays (row_ptr, col, val, b) of the RCS at the scene's initial
    values and the library's initial damping 1e-4."""
    s = _scene(case, seed)
    n, lam = case["n"], 1e-4
    e, Jc, Jp, _ = _linearize(s, s["cams"], s["pts"], None, None, 0.0)
    oc, op = s["oc"], s["op"]
    V = _segsum((Jp.transpose(1, 2) @ Jp).flatten(1), op)[0].view(-1, 3, 3)
    V = V + lam * torch.diag_embed(V.diagonal(dim1=1, dim2=2).clamp(1e-6, 1e32))
    lp = _segsum(-(Jp * e[:, :, None]).sum(1), op)[0]
    Vi = torch.linalg.inv(V)
    A = Jc.transpose(1, 2) @ Jp  # W
    U = _segsum((Jc.transpose(1, 2) @ Jc).flatten(1), oc)[0].view(-1, 6, 6)
    lc = _segsum(-(Jc * e[:, :, None]).sum(1), oc)[0]
    AV = A @ Vi[op]
    b = lc - _segsum((AV @ lp[op][:, :, None])[:, :, 0], oc)[0]
    # ordered pairs (a <= b) of the observations of a point
    cnt = torch.bincount(op)
    start = torch.cumsum(cnt, 0) - cnt
    pa, pb = [], []
    for d in range(int(cnt.max())):
        i = torch.nonzero(torch.arange(len(op), device=DEV) - start[op] + d < cnt[op])[:, 0]
        pa.append(i)
        pb.append(i + d)
    pa, pb = torch.cat(pa), torch.cat(pb)
    S, key = _segsum(-(AV[pa] @ A[pb].transpose(1, 2)).flatten(1), oc[pa] * n + oc[pb])
    S = S.view(-1, 6, 6)
    row, col = key // n, key % n
    d = row == col
    S[d] = S[d] + U + lam * torch.diag_embed(U.diagonal(dim1=1, dim2=2).clamp(1e-6, 1e32))
    S[d] = 0.5 * (S[d] + S[d].transpose(1, 2))
    row_ptr = torch.zeros(n + 1, dtype=torch.int32, device=DEV)
    row_ptr[1:] = torch.cumsum(torch.bincount(row, minlength=n), 0)
    return row_ptr, col.to(torch.int32), S.float(), b.float()


def _grid_pattern(n, nl):
    """Upper block pattern of a nadir grid: each camera and its neighbours up
    to four along and two across."""
    k = torch.arange(n, device=DEV)
    ix = k % nl
    rows, cols = [k], [k]
    for dj in range(0, 3):
        for di in range(-4, 5):
            if dj == 0 and di <= 0:
                continue
            m = (ix + di >= 0) & (ix + di < nl) & (k + dj * nl + di < n)
            rows.append(k[m])
            cols.append(k[m] + dj * nl + di)
    key, _ = torch.sort(torch.cat(rows) * n + torch.cat(cols))
    return key // n, key % n


def _vb_system(case, seed):
    """Variable-size SPD system on the grid pattern: N(0, 1) off-diagonal
    values, and diagonal blocks G G^T / c + t I with t a little above the
    norm of the off-diagonal part (PCG takes a few tens of iterations); the
    blocks as nnzb x 11 x 11 (zero beyond c_i x c_j)."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed * 104729 + 5)
    n = case["n"]
    row, col = _grid_pattern(n, case["along"])
    # which cameras carry interiors belongs to the case, spread over the grid
    c = torch.where(torch.frac(0.618034 * torch.arange(n, device=DEV, dtype=F64)) < case["frac"], 11, 6)
    live = torch.arange(11, device=DEV)[None] < c[:, None]
    S = torch.randn(len(row), 11, 11, generator=g, device=DEV, dtype=F64)
    S = S * (live[row][:, :, None] & live[col][:, None, :])
    d = row == col
    sq = torch.where(d, torch.zeros((), device=DEV, dtype=F64), S.flatten(1).square().sum(1))[:, None]
    t = 2.2 * ((_segsum(sq, row)[0] + _segsum(sq, col)[0])[:, 0] / c).max().sqrt()
    D = S[d] @ S[d].transpose(1, 2) / c[:, None, None] + t * torch.diag_embed(live.to(F64))
    S[d] = 0.5 * (D + D.transpose(1, 2))
    b = torch.randn(n, 11, generator=g, device=DEV, dtype=F64) * live
    if case["fp32"]:
        S, b = S.float().to(F64), b.float().to(F64)
    x = torch.randn(n, 11, generator=g, device=DEV, dtype=F64) * live
    return row, col, c, live, S, b, x.float().to(F64)


# ---------------------------------------------------------------------------
# the measured calls
# ---------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind in ("solve", "static"):
        rp, col, val, b = _schur_system(case, seed)
        if kind == "solve":
            st["p"] = B.Problem.from_rcs(_host(rp), _host(col), _host(val, np.float64), _host(b, np.float64),
                                         precision=B.BA_FP32, pcg_rel_tol=case["tol"])
        else:
            st.update(rp=rp, col=col, val=val.contiguous(), b=b.contiguous(), x=torch.empty_like(b))
        return st
    prec = B.BA_FP32 if case["fp32"] else B.BA_FP64
    T = torch.float32 if case["fp32"] else F64
    if kind == "vbsmc":
        row, col, c, live, S, b, x = _vb_system(case, seed)
        n = case["n"]
        rp = np.zeros(n + 1, np.int32)
        rp[1:] = _host(torch.cumsum(torch.bincount(row, minlength=n), 0))
        mask = live[row][:, :, None] & live[col][:, None, :]
        st["p"] = B.VBSMC(_host(c, np.int32), rp, _host(col, np.int32), _host(S[mask]), _host(b[live]), precision=prec)
        st["x"] = x[live].to(T)
        st["y"] = torch.empty_like(st["x"])
        return st
    s = _scene(case, seed)
    obs = (_host(s["oc"], np.int32), _host(s["op"], np.int64), _host(s["uv"]))
    st["cams"], st["pts"] = _pinned(s["cams"]), _pinned(s["pts"])
    if kind == "interiors":
        st["intr"] = _pinned(s["intr"])
        st["p"] = B.VBIProblem(st["cams"], st["intr"], _host(s["cdim"]), st["pts"], *obs, precision=prec,
                               pcg_rel_tol=case["tol"])
        return st
    st["p"] = B.Problem(st["cams"], st["pts"], *obs, precision=prec, pcg_rel_tol=case.get("tol", 1e-10),
                        robust=B.BA_LOSS_HUBER if case["huber"] else B.BA_LOSS_PLAIN)
    if kind == "form":
        g = torch.Generator(device=DEV)
        g.manual_seed(seed + 3)
        st["x"] = torch.randn(6 * case["n"], generator=g, device=DEV, dtype=F64).float().to(T)
        st["y"] = torch.empty_like(st["x"])
    else:
        st["cams_out"] = _pinned(s["cams"])
        st["pts_out"] = _pinned(s["pts"])
    return st


def _given(case, a):
    """A result array in the problem's precision."""
    return torch.from_numpy(a).float() if case["fp32"] else torch.from_numpy(a)


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "lm":
        p = st["p"]
        p.set_state(st["cams"], st["pts"], 1e-4)
        for _ in range(case["steps"]):
            info = p.lm_step()
        cams = B.ba_get_cameras(p.h, p.n, st["cams_out"])
        pts = B.ba_get_points(p.h, p.P, st["pts_out"])
        return {"cams": _given(case, cams), "pts": _given(case, pts), "cost": info["cost_after"],
                "accepted": info["accepted"]}
    if kind == "interiors":
        p = st["p"]
        p.set_state(st["cams"], st["intr"], st["pts"], case["lam"], 2.0)
        for _ in range(case["steps"]):
            info = p.lm_step()
        cams, intr, pts = p.state()
        return {"cams": _given(case, cams), "intr": _given(case, intr), "pts": _given(case, pts),
                "cost": info["cost_after"], "accepted": info["accepted"]}
    if kind == "form":
        p = st["p"]
        cost = p.linearize()
        p.form_rcs(1e-4)
        p.rcs_spmv(B.BA_FMT_BSMC, st["x"], st["y"])
        return {"y": st["y"], "cost": cost}
    if kind == "solve":
        st["p"].solve_rcs()
        return {"x": torch.from_numpy(st["p"].step()[0]).float()}
    if kind == "static":
        B.ba_pcg_solve_static(case["n"], len(st["col"]), st["rp"].data_ptr(), st["col"].data_ptr(),
                              st["val"].data_ptr(), st["b"].data_ptr(), st["x"].data_ptr(), case["tol"], 0,
                              torch.cuda.current_stream().cuda_stream)
        return {"x": st["x"]}
    st["p"].spmv(st["x"], st["y"])
    x = st["p"].solve(case["tol"])[0]
    return {"y": st["y"], "x": _given(case, x)}


def work(case):
    """Inputs read once and results written once; FMAs of the formation (one
    product of two observations of a track is 12 + 2 c + 2 c c FMAs, about 18
    products per point) or of one product with the system."""
    n, e = case["n"], 8 if case.get("fp32") is False else 4
    if case["kind"] == "vbsmc":
        cc = (11 * case["frac"] + 6 * (1 - case["frac"])) ** 2
        return {"bytes": 23 * n * cc * e, "flops": 2 * 45 * n * cc}
    if case["kind"] in ("solve", "static"):
        nb = (20 if n < 100 else 32) * n
        return {"bytes": nb * 148 + 48 * n, "flops": 2 * 72 * nb}
    c = 6 + 5 * case.get("frac", 0.0)
    obs, P = 5 * case["pts"], case["pts"]
    steps = case.get("steps", 1)
    state = (6 * n + 3 * P + (5 * n if case["kind"] == "interiors" else 0)) * 8
    return {"bytes": obs * (8 + 2 * e) + 2 * state, "flops": steps * P * 18 * 2 * (12 + 2 * c + 2 * c * c)}


# ---------------------------------------------------------------------------
# the same results in 64 bits, by plain torch
# ---------------------------------------------------------------------------

def _cost(s, cams, pts, intr, delta):
    oc, op = s["oc"], s["op"]
    Xc = torch.einsum("mij,mj->mi", _qrot(_qexp(cams[:, :3]))[oc], pts[op]) + cams[oc, 3:]
    e = _project(Xc, None if intr is None else intr[oc])[0] - s["uv"]
    q = e.square().sum(1)
    if delta:
        q = torch.where(q > delta * delta, 2 * delta * q.sqrt() - delta * delta, q)
    return float(0.5 * q.sum())


def _project(Xc, k):
    h = Xc[:, :2] / Xc[:, 2:]
    if k is None:
        return F * h + C, h, None, None
    r2 = h.square().sum(1, keepdim=True)
    d = 1 + k[:, 3:4] * r2 + k[:, 4:5] * r2 * r2
    return k[:, :1] * d * h + k[:, 1:3], h, r2, d


def _linearize(s, cams, pts, intr, cdim, delta):
    """e (m x 2), J_c (m x 2 x c), J_p (m x 2 x 3) and the cost."""
    oc, op = s["oc"], s["op"]
    R = _qrot(_qexp(cams[:, :3]))[oc]
    Xc = torch.einsum("mij,mj->mi", R, pts[op]) + cams[oc, 3:]
    k = None if intr is None else intr[oc]
    u, h, r2, d = _project(Xc, k)
    e = u - s["uv"]
    m = len(oc)
    dh = torch.zeros(m, 2, 3, device=DEV, dtype=F64)  # d(x/z, y/z) / dX_cam
    dh[:, 0, 0] = dh[:, 1, 1] = 1 / Xc[:, 2]
    dh[:, :, 2] = -h / Xc[:, 2:]
    if k is None:
        Jx = F * dh
    else:
        g = (2 * k[:, 3:4] + 4 * k[:, 4:5] * r2)[:, :, None]
        D = k[:, :1, None] * (d[:, :, None] * torch.eye(2, device=DEV, dtype=F64) + g * h[:, :, None] * h[:, None, :])
        Jx = D @ dh
    X0, X1, X2 = Xc.unbind(1)
    o = torch.zeros_like(X0)
    M = torch.stack([o, X2, -X1, -X2, o, X0, X1, -X0, o], 1).view(m, 3, 3)
    Jc = [Jx @ M, Jx]
    if k is not None:
        J5 = torch.zeros(m, 2, 5, device=DEV, dtype=F64)
        J5[:, :, 0] = d * h
        J5[:, 0, 1] = J5[:, 1, 2] = 1
        J5[:, :, 3] = k[:, :1] * r2 * h
        J5[:, :, 4] = k[:, :1] * r2 * r2 * h
        Jc.append(J5 * (cdim[oc] == 11)[:, None, None])
    Jc, Jp = torch.cat(Jc, 2), Jx @ R
    q = e.square().sum(1)
    rho = q
    if delta:
        bent = q > delta * delta
        rho = torch.where(bent, 2 * delta * q.sqrt() - delta * delta, q)
        w = torch.where(bent, (delta / q.sqrt().clamp_min(1e-300)).sqrt(), torch.ones_like(q))
        e, Jc, Jp = e * w[:, None], Jc * w[:, None, None], Jp * w[:, None, None]
    return e, Jc, Jp, float(0.5 * rho.sum())


class _Schur:
    """The damped RCS of a linearization, applied without being stored."""

    def __init__(self, s, n, P, e, Jc, Jp, lam, cdim):
        self.oc, self.op, self.n, self.P, self.Jc, self.Jp = s["oc"], s["op"], n, P, Jc, Jp
        c = Jc.shape[2]

        def sum_c(x):
            return torch.zeros(n, *x.shape[1:], device=DEV, dtype=F64).index_add_(0, self.oc, x)

        def sum_p(x):
            return torch.zeros(P, *x.shape[1:], device=DEV, dtype=F64).index_add_(0, self.op, x)

        self.sum_c, self.sum_p = sum_c, sum_p
        V = sum_p(Jp.transpose(1, 2) @ Jp)
        V = V + lam * torch.diag_embed(V.diagonal(dim1=1, dim2=2).clamp(1e-6, 1e32))
        self.Vi = torch.linalg.inv(V)
        self.lp = -sum_p((Jp * e[:, :, None]).sum(1))
        U = sum_c(Jc.transpose(1, 2) @ Jc)
        dg = U.diagonal(dim1=1, dim2=2)
        self.damp = lam * dg.clamp(1e-6, 1e32)
        if cdim is not None and c == 11:
            self.fixed = (cdim != 11)[:, None] & (torch.arange(11, device=DEV) >= 6)
            self.damp = torch.where(self.fixed, torch.ones_like(dg), self.damp)
        W = Jc.transpose(1, 2) @ Jp
        self.b = -sum_c((Jc * e[:, :, None]).sum(1)) - sum_c((W @ (self.Vi @ self.lp[:, :, None])[self.op])[:, :, 0])
        self.M = torch.linalg.inv(U + torch.diag_embed(self.damp) - sum_c(W @ self.Vi[self.op] @ W.transpose(1, 2)))

    def Jx(self, x):
        return (self.Jc @ x[self.oc][:, :, None])[:, :, 0]

    def points(self, dc, lp):
        t = self.sum_p((self.Jp * self.Jx(dc)[:, :, None]).sum(1))
        return (self.Vi @ (lp - t)[:, :, None])[:, :, 0]

    def apply(self, x):
        v = self.Jx(x)
        w = self.points(x, 0.0)
        v = v + (self.Jp @ w[self.op][:, :, None])[:, :, 0]
        return self.sum_c((self.Jc * v[:, :, None]).sum(1)) + self.damp * x


def _pcg(apply, M, b, tol, most=20000):
    x, r = torch.zeros_like(b), b.clone()
    z = (M @ r[:, :, None])[:, :, 0]
    d, rz, r0 = z, (r * z).sum(), r.norm()
    for _ in range(most):
        q = apply(d)
        a = rz / (d * q).sum()
        x = x + a * d
        r = r - a * q
        if r.norm() <= tol * r0:
            break
        z = (M @ r[:, :, None])[:, :, 0]
        new = (r * z).sum()
        d, rz = z + (new / rz) * d, new
    return x


def _block_apply(row, col, S):
    off = row != col

    def apply(x):
        y = torch.zeros_like(x).index_add_(0, row, (S @ x[col][:, :, None])[:, :, 0])
        return y.index_add_(0, col[off], (S[off].transpose(1, 2) @ x[row[off]][:, :, None])[:, :, 0])
    return apply


def exact(case, seed):
    kind = case["kind"]
    if kind in ("solve", "static"):
        rp, col, S, b = _schur_system(case, seed)
        row = torch.repeat_interleave(torch.arange(case["n"], device=DEV), torch.diff(rp.long()))
        col, S, b = col.long(), S.to(F64), b.to(F64)
        x = _pcg(_block_apply(row, col, S), torch.linalg.inv(S[row == col]), b, 1e-14, 40 * case["n"] + 500)
        return {"x": x.flatten().view(-1, 6)}
    if kind == "vbsmc":
        row, col, c, live, S, b, x = _vb_system(case, seed)
        apply = _block_apply(row, col, S)
        D = S[row == col] + torch.diag_embed((~live).to(F64))
        return {"y": apply(x)[live], "x": _pcg(apply, torch.linalg.inv(D), b, 1e-15, 500)[live]}
    s = _scene(case, seed)
    cams, pts, intr, cdim = s["cams"], s["pts"], s.get("intr"), s.get("cdim")
    n, P, delta = case["n"], len(pts), 2.0 if case.get("huber") else 0.0
    if kind == "form":
        e, Jc, Jp, cost = _linearize(s, cams, pts, None, None, delta)
        g = torch.Generator(device=DEV)
        g.manual_seed(seed + 3)
        x = torch.randn(6 * n, generator=g, device=DEV, dtype=F64).float().to(F64)
        return {"y": _Schur(s, n, P, e, Jc, Jp, 1e-4, None).apply(x.view(n, 6)).flatten(), "cost": cost}
    lam, nu = case.get("lam", 1e-4), 2.0
    for _ in range(case["steps"]):
        e, Jc, Jp, cost = _linearize(s, cams, pts, intr, cdim, delta)
        A = _Schur(s, n, P, e, Jc, Jp, lam, cdim)
        dc = _pcg(A.apply, A.M, A.b, case["tol"])
        dp = A.points(dc, A.lp)
        Jd = A.Jx(dc) + (Jp @ dp[A.op][:, :, None])[:, :, 0]
        pred = float(-0.5 * (Jd * (2 * e + Jd)).sum())
        qd = _qexp(dc[:, :3])
        c1 = torch.cat([_qlog(_qmul(qd, _qexp(cams[:, :3]))),
                        (_qrot(qd) @ cams[:, 3:, None])[:, :, 0] + dc[:, 3:6]], 1)
        p1 = pts + dp
        i1 = None if intr is None else intr + torch.where((cdim == 11)[:, None], dc[:, 6:], 0.0)
        F1 = _cost(s, c1, p1, i1, delta)
        rho = (cost - F1) / pred
        if pred > 0 and rho > 1e-3:
            cams, pts, intr, cost, took = c1, p1, i1, F1, 1
            lam, nu = lam * max(1 / 3, 1 - (2 * rho - 1) ** 3), 2.0
        else:
            took, lam, nu = 0, lam * nu, 2 * nu
    out = {"cams": cams, "pts": pts, "cost": cost, "accepted": None}
    if intr is not None:
        out["intr"] = intr
    return out
