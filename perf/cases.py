"""Performance cases of the optimiser: what programs that use the library have it do.

Every pass goes through the binding's public entry points.  A solve pass writes the
initial state into a resident graph, runs Levenberg-Marquardt iterations and reads the
optimised state back, all on device buffers, as a back end does whenever its front end
hands it a new estimate.  Scenes come from the package's seeded generators at the sizes
of its tests, its benchmark and its served windows.

The LM iterations of the path scenes start from a damping of 0.01 to 0.3, where Nielsen's
rule has taken it when steps are first accepted there (the default 1e-4 overshoots on
them), so that every pass ends in a changed state.

With FP32 or BF16 storage the linear system, and with it every step, carries FP32's
accuracy; such a program keeps its map in FP32 (as rendering and mapping code does), so
those cases return the state and the final cost as float32.  The FP64 cases return what
the library wrote, as float64.
"""
import ctypes
import dataclasses
import math

import numpy as np
import torch

from paper_2509_26581_gb300 import gpo, serving, synth

DEV = "cuda"


def listed():
    return [
        # the smallest solve: a 10-camera problem refined in place (calibration rigs, tests)
        dict(name="ring_small_fp64", kind="ba", scene="ring", cams=10, pts=500, views=6, robust=False,
             prec="fp64", iters=10, damping=1e-4, solver="schur"),
        # local bundle adjustment of a SLAM back end: one window, first keyframe fixed
        dict(name="window_bf16", kind="ba", scene="window", cams=20, pts=2000, prec="bf16", iters=2,
             damping=0.1, solver="schur"),
        # many sessions' windows of different sizes solved together
        dict(name="windows_batch_bf16", kind="batch", windows=24, kf_lo=5, kf_hi=40, pts_lo=300, pts_hi=8000,
             prec="bf16", iters=2, damping=0.1),
        # wide-baseline reconstruction (100 cameras, 300,000 observations, outliers)
        dict(name="ring_mid_fp32", kind="ba", scene="ring", cams=100, pts=50_000, views=6, robust=True,
             prec="fp32", iters=3, damping=1e-4, solver="schur"),
        # mapping run where FP64 is asked for throughout
        dict(name="path_fp64", kind="ba", scene="path", cams=300, pts=100_000, law="pareto", prec="fp64",
             iters=1, damping=0.1, solver="schur"),
        # a mapping run of odd sizes, FP32 storage
        dict(name="path_odd_fp32", kind="ba", scene="path", cams=777, pts=250_001, law="pareto", prec="fp32",
             iters=1, damping=0.01, solver="schur"),
        # the benchmark's workload (1,000 cameras, 500,000 points, 3M observations), BF16 storage
        dict(name="path_medium_bf16", kind="ba", scene="path", cams=1000, pts=500_000, law="pareto", prec="bf16",
             iters=2, damping=0.1, solver="schur"),
        # a long mapping run with geometric track lengths: the largest
        dict(name="path_large_bf16", kind="ba", scene="path", cams=4000, pts=1_400_000, law="geom", prec="bf16",
             iters=1, damping=0.3, solver="schur"),
        # a visual-inertial window, FP64
        dict(name="vi_window_fp64", kind="vi", kfs=20, pts=1500, prec="fp64", iters=2, damping=0.01),
        # global visual-inertial adjustment of a session, BF16 storage
        dict(name="vi_session_bf16", kind="vi", kfs=1000, pts=66_000, prec="bf16", iters=1, damping=0.01),
        # the paper's own linear system: cameras and points together
        dict(name="full_system_fp32", kind="ba", scene="ring", cams=60, pts=20_000, views=6, robust=True,
             prec="fp32", iters=2, damping=1e-4, solver="full"),
        # the cost of a state on caller-owned buffers, from a thread that must not allocate
        dict(name="cost_fp64", kind="cost", cams=400, pts=165_000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["ring", "ring", "path", "path", "path", "window", "batch", "vi", "vi", "full", "cost"])
    prec = rng.choice(["fp64", "fp32", "bf16"])
    if kind in ("ring", "full"):
        cams = _log(rng, 8, 128)
        return dict(kind="ba", scene="ring", cams=cams, pts=_log(rng, 300, 60_000 if kind == "ring" else 25_000),
                    views=rng.randint(4, min(12, cams)), robust=rng.random() < 0.5, prec=prec,
                    iters=rng.randint(1, 3), damping=1e-4, solver="schur" if kind == "ring" else "full")
    if kind == "path":
        cams = _log(rng, 40, 1500)
        pts = min(cams * rng.randint(60, 500), 150_000 if prec == "fp64" else 500_000) + rng.randint(0, 99)
        iters = rng.randint(1, 2)
        return dict(kind="ba", scene="path", cams=cams, pts=pts, law=rng.choice(["pareto", "geom"]), prec=prec,
                    iters=iters, damping=0.1 if iters > 1 else rng.choice([0.1, 0.01]), solver="schur")
    if kind == "window":
        return dict(kind="ba", scene="window", cams=rng.randint(5, 40), pts=_log(rng, 300, 8000), prec=prec,
                    iters=2, damping=0.1, solver="schur")
    if kind == "batch":
        return dict(kind="batch", windows=rng.randint(2, 40), kf_lo=5, kf_hi=rng.randint(8, 40), pts_lo=300,
                    pts_hi=_log(rng, 1000, 8000), prec=prec, iters=2, damping=0.1)
    if kind == "vi":
        kfs = _log(rng, 8, 800)
        return dict(kind="vi", kfs=kfs, pts=kfs * rng.randint(50, 90) + rng.randint(0, 9), prec=prec, iters=1,
                    damping=0.01)
    return dict(kind="cost", cams=_log(rng, 20, 500), pts=_log(rng, 2000, 250_000))


# ---------------------------------------------------------------- inputs

def _first(p, n, cam):
    """The scene's first n points with their observations (the generators drop points that
    fewer than two views see, so they are asked for more than n)."""
    if p.n_pts < n:
        raise ValueError("the scene has %d points, %d are wanted" % (p.n_pts, n))
    keep = p.pt_idx < n
    return dataclasses.replace(p, pts_gt=p.pts_gt[:n], pts0=p.pts0[:n], pt_idx=p.pt_idx[keep], obs=p.obs[keep],
                               **{cam: getattr(p, cam)[keep]}, **({} if cam == "kf_idx" else dict(is_outlier=p.is_outlier[keep])))


def _path(seed, cams, pts, law="pareto"):
    spare = 2 * pts if cams < 12 else pts if cams < 24 else pts // 4 if cams < 48 else pts // 50
    return _first(synth.ba_path(seed, cams, pts + spare + 8, law), pts, "cam_idx")


def _vi(case, seed):
    pts = case["pts"]
    return _first(synth.vi_problem(seed, case["kfs"], pts + pts // 8 + 16), pts, "kf_idx")


def _windows(case, seed):
    """The batch's windows: sizes by the case alone, scenes by the seed."""
    rng = synth.Stream(case["windows"], 21)
    kf = rng.integers(case["windows"], case["kf_lo"], case["kf_hi"] + 1)
    pts = rng.integers(case["windows"], case["pts_lo"], case["pts_hi"] + 1)
    return [_path(seed * 1000003 + i, int(k), int(n)) for i, (k, n) in enumerate(zip(kf, pts))]


def _scene(case, seed):
    if case["kind"] == "cost":
        return _path(seed, case["cams"], case["pts"])
    if case["scene"] == "ring":
        kw = dict(outlier_frac=0.01, huber_delta=2.0) if case["robust"] else {}
        return synth.ba_ring(seed, case["cams"], case["pts"], case["views"], **kw)
    return _path(seed, case["cams"], case["pts"], case.get("law", "pareto"))


def _params(case):
    kw = dict(initial_damping=case["damping"])
    if case["kind"] == "vi":
        kw["pcg_rejection_ratio"] = 0.0       # the inertial chain's residual rises before it falls
    if case.get("solver") == "full":
        kw["solver"] = gpo.GPO_SOLVER_FULL
    return gpo.default_params(**kw)


def _dev(a, dtype=None):
    t = torch.from_numpy(np.ascontiguousarray(a)).to(DEV)
    return t if dtype is None else t.to(dtype)


def _resident(g, c0, p0, cams, pts):
    """A graph on the device with its initial state and the buffers its result is read into."""
    g.optimize(0)
    cd, pd = _dev(cams), _dev(pts)
    return dict(g=g, c0=c0, p0=p0, cams=cd, pts=pd, cams_out=torch.empty_like(cd), pts_out=torch.empty_like(pd))


def prepare(case, seed):
    st = dict(case=case)
    if case["kind"] == "cost":
        p = _scene(case, seed)
        st.update(cams=_dev(p.cams0), pts=_dev(p.pts0), cam=_dev(p.cam_idx), pt=_dev(p.pt_idx), obs=_dev(p.obs),
                  delta=float(p.huber_delta), out=torch.empty(1, dtype=torch.float64, device=DEV))
        return st
    st["params"] = _params(case)
    if case["kind"] == "vi":
        p = _vi(case, seed)
        g, n0, p0, _ = gpo.vi_graph(p, precision=case["prec"])
        st["parts"] = [_resident(g, n0, p0, p.nav0, p.pts0)]
    elif case["kind"] == "batch":
        st["parts"] = [_resident(*serving.window_graph(p, case["prec"]), p.cams0, p.pts0)
                       for p in _windows(case, seed)]
    else:
        p = _scene(case, seed)
        if case["scene"] == "window":
            g, c0, p0 = serving.window_graph(p, case["prec"])
        else:
            g, c0, p0 = gpo.ba_graph(p.cams0, p.pts0, p.cam_idx, p.pt_idx, p.obs, p.huber_delta, case["prec"])
        st["parts"] = [_resident(g, c0, p0, p.cams0, p.pts0)]
    return st


# ---------------------------------------------------------------- one pass

def run(st):
    case = st["case"]
    if case["kind"] == "cost":
        s = gpo.lib.gpo_ba_cost_noalloc(torch.cuda.current_device(),
                                        ctypes.c_void_p(torch.cuda.current_stream().cuda_stream),
                                        ctypes.c_void_p(st["cams"].data_ptr()), ctypes.c_void_p(st["pts"].data_ptr()),
                                        ctypes.c_void_p(st["cam"].data_ptr()), ctypes.c_void_p(st["pt"].data_ptr()),
                                        ctypes.c_void_p(st["obs"].data_ptr()), st["cam"].shape[0], st["delta"],
                                        ctypes.c_void_p(st["out"].data_ptr()))
        if s != gpo.GPO_OK:
            raise RuntimeError("gpo_ba_cost_noalloc: status %d" % s)
        return st["out"]
    parts = st["parts"]
    for q in parts:
        q["g"].set_initial(q["c0"], q["cams"])
        q["g"].set_initial(q["p0"], q["pts"])
    if case["kind"] == "batch":
        reps = gpo.optimize_batch([q["g"] for q in parts], case["iters"], st["params"])
    else:
        reps = [parts[0]["g"].optimize(case["iters"], st["params"])]
    for q in parts:
        q["g"].get_state(q["c0"], q["cams"].shape[0], q["cams"].shape[1], out=q["cams_out"])
        q["g"].get_state(q["p0"], q["pts"].shape[0], 3, out=q["pts_out"])
    if case["kind"] == "batch":   # the sessions' maps one after another
        cams, pts = (torch.cat([q[k] for q in parts]) for k in ("cams_out", "pts_out"))
    else:
        cams, pts = parts[0]["cams_out"], parts[0]["pts_out"]
    first = np.array([r.initial_cost for r in reps])
    last = np.array([r.final_cost for r in reps])
    if case["prec"] != "fp64":
        cams, pts, last = cams.float(), pts.float(), last.astype(np.float32)
    return dict(cams=cams, pts=pts, initial_cost=first, final_cost=last)


def work(case):
    """Bytes: measurements and indices read once, states read and written once.  Flops: per
    LM iteration the rows, normal-equation blocks and two costs of every observation."""
    if case["kind"] == "batch":
        cams, pts = case["windows"] * (case["kf_lo"] + case["kf_hi"]) / 2, case["windows"] * (case["pts_lo"] + case["pts_hi"]) / 2
    else:
        cams, pts = case.get("cams", case.get("kfs")), case["pts"]
    views = case.get("views") or (9.5 if case["kind"] == "vi" else 6.4 if case.get("law") == "geom" else 5.9)
    edges = pts * views
    if case["kind"] == "cost":
        return dict(bytes=edges * 24 + pts * 24 + cams * 72, flops=edges * 70)
    vi = case["kind"] == "vi"
    return dict(bytes=edges * (32 if vi else 24) + 2 * (pts * 24 + cams * (128 if vi else 72)),
                flops=case["iters"] * edges * (1100 if vi else 900))


# ---------------------------------------------------------------- the same in 64 bits, plain torch
#
# Levenberg-Marquardt with Nielsen's damping; each step by block-Jacobi PCG (relative
# tolerance 1e-6, at most 100 iterations) on the camera Schur complement or on the full
# system, with matrix-free products of explicit Jacobians; Jacobians by forward-mode
# differentiation on the update chart.

G = (0.0, 0.0, -9.81)


def _cross(a, b):
    return torch.linalg.cross(a, b)


def _hat(w):
    z = torch.zeros_like(w[..., 0])
    return torch.stack([z, -w[..., 2], w[..., 1], w[..., 2], z, -w[..., 0], -w[..., 1], w[..., 0], z], -1).reshape(
        w.shape[:-1] + (3, 3))


def _so3(w):
    """Rodrigues' formula; below an angle of 1e-6 the series."""
    t2 = (w * w).sum(-1, keepdim=True)[..., None]
    small = t2 < 1e-12
    t = torch.sqrt(torch.where(small, torch.ones_like(t2), t2))
    a = torch.where(small, 1 - t2 / 6, torch.sin(t) / t)
    b = torch.where(small, 0.5 - t2 / 24, (1 - torch.cos(t)) / (t * t))
    K = _hat(w)
    return torch.eye(3, dtype=w.dtype, device=w.device) + a * K + b * (K @ K)


def _log3(R):
    v = 0.5 * torch.stack([R[..., 2, 1] - R[..., 1, 2], R[..., 0, 2] - R[..., 2, 0], R[..., 1, 0] - R[..., 0, 1]], -1)
    s = torch.sqrt((v * v).sum(-1, keepdim=True) + 1e-300)
    c = 0.5 * (R[..., 0, 0] + R[..., 1, 1] + R[..., 2, 2] - 1)[..., None]
    return v * torch.where(s < 1e-9, torch.ones_like(s), torch.atan2(s, c) / s)


def _quat(w):
    t = torch.linalg.vector_norm(w, dim=-1, keepdim=True)
    k = torch.where(t < 1e-9, 0.5 * torch.ones_like(t), torch.sin(0.5 * t) / torch.where(t < 1e-9, torch.ones_like(t), t))
    return torch.cat([w * k, torch.cos(0.5 * t)], -1)                      # x y z w


def _qmul(a, b):
    av, aw, bv, bw = a[..., :3], a[..., 3:], b[..., :3], b[..., 3:]
    return torch.cat([aw * bv + bw * av + _cross(av, bv), aw * bw - (av * bv).sum(-1, keepdim=True)], -1)


def _qrot(q):
    q = q / torch.linalg.vector_norm(q, dim=-1, keepdim=True)
    v, w = q[..., :3], q[..., 3:, None]
    K = _hat(v)
    return torch.eye(3, dtype=q.dtype, device=q.device) + 2 * w * K + 2 * (K @ K)


def _ba_residual(d, cam, R, X, z):
    """Reprojection at the state moved by d = [dw dt df dk1 dk2 dX] (first order in dw)."""
    y = R @ (X + d[9:12])
    P = y + _cross(d[0:3], y) + cam[3:6] + d[3:6]
    p = -P[:2] / P[2]
    q = (p * p).sum()
    return (cam[6] + d[6]) * (1 + (cam[7] + d[7]) * q + (cam[8] + d[8]) * q * q) * p - z


def _stereo_residual(d, nav, R, X, z, rig):
    y = R.T @ (X + d[6:9] - nav[4:7] - R @ d[3:6])
    Xc = rig["R"] @ (y - _cross(d[0:3], y)) + rig["t"]
    return torch.stack([rig["fx"] * Xc[0] / Xc[2] + rig["cx"], rig["fy"] * Xc[1] / Xc[2] + rig["cy"],
                        rig["fx"] * (Xc[0] - rig["b"]) / Xc[2] + rig["cx"]]) - z


def _imu_residual(d, xi, xj, Ri, Rj, m):
    g = torch.tensor(G, dtype=xi.dtype, device=xi.device)
    Ri1, Rj1 = Ri + Ri @ _hat(d[0:3]), Rj + Rj @ _hat(d[15:18])
    pi, pj = xi[4:7] + Ri @ d[3:6], xj[4:7] + Rj @ d[18:21]
    vi, vj = xi[7:10] + d[6:9], xj[7:10] + d[21:24]
    dbg, dba = xi[10:13] + d[9:12] - m["bg0"], xi[13:16] + d[12:15] - m["ba0"]
    T = m["T"]
    return torch.cat([_log3((m["dR"] @ _so3(m["JRg"] @ dbg)).T @ Ri1.T @ Rj1),
                      Ri1.T @ (vj - vi - g * T) - (m["dv"] + m["Jvg"] @ dbg + m["Jva"] @ dba),
                      Ri1.T @ (pj - pi - vi * T - 0.5 * g * T * T) - (m["dp"] + m["Jpg"] @ dbg + m["Jpa"] @ dba)])


def _preintegrate(p):
    """On-manifold preintegration of every keyframe interval at the initial biases (batched)."""
    w, a = _dev(p.imu_gyro), _dev(p.imu_acc)
    K, N, dt = w.shape[0], w.shape[1], p.dt
    bg0, ba0 = _dev(p.nav0[:-1, 10:13]), _dev(p.nav0[:-1, 13:16])
    eye = torch.eye(3, dtype=torch.float64, device=DEV).expand(K, 3, 3)
    z3 = torch.zeros(K, 3, 3, dtype=torch.float64, device=DEV)
    dR, dv, dp = eye.clone(), z3[:, 0].clone(), z3[:, 0].clone()
    JRg, Jvg, Jva, Jpg, Jpa = (z3.clone() for _ in range(5))
    cov = torch.zeros(K, 9, 9, dtype=torch.float64, device=DEV)
    qg, qa = p.noise["sigma_g"] ** 2 / dt, p.noise["sigma_a"] ** 2 / dt
    for k in range(N):
        phi, acc = (w[:, k] - bg0) * dt, a[:, k] - ba0
        dRk, h = _so3(phi), _hat(acc)
        t2 = (phi * phi).sum(-1)[:, None, None]
        t = torch.sqrt(t2 + 1e-300)
        small = t2 < 1e-12
        Kp = _hat(phi)
        Jr = (torch.eye(3, dtype=torch.float64, device=DEV)
              - torch.where(small, 0.5 - t2 / 24, (1 - torch.cos(t)) / t2.clamp_min(1e-300)) * Kp
              + torch.where(small, 1 / 6 - t2 / 120, (t - torch.sin(t)) / (t2 * t).clamp_min(1e-300)) * (Kp @ Kp))
        A = torch.eye(9, dtype=torch.float64, device=DEV).repeat(K, 1, 1)
        A[:, 0:3, 0:3] = dRk.transpose(1, 2)
        A[:, 3:6, 0:3] = -dR @ h * dt
        A[:, 6:9, 0:3] = -0.5 * dR @ h * dt * dt
        A[:, 6:9, 3:6] = eye * dt
        Bg, Ba = torch.zeros(K, 9, 3, dtype=torch.float64, device=DEV), torch.zeros(K, 9, 3, dtype=torch.float64, device=DEV)
        Bg[:, 0:3] = Jr * dt
        Ba[:, 3:6] = dR * dt
        Ba[:, 6:9] = 0.5 * dR * dt * dt
        cov = A @ cov @ A.transpose(1, 2) + qg * Bg @ Bg.transpose(1, 2) + qa * Ba @ Ba.transpose(1, 2)
        Jpa = Jpa + Jva * dt - 0.5 * dR * dt * dt
        Jpg = Jpg + Jvg * dt - 0.5 * dR @ h @ JRg * dt * dt
        Jva = Jva - dR * dt
        Jvg = Jvg - dR @ h @ JRg * dt
        JRg = dRk.transpose(1, 2) @ JRg - Jr * dt
        Ra = (dR @ acc[:, :, None])[:, :, 0]
        dp = dp + dv * dt + 0.5 * Ra * dt * dt
        dv = dv + Ra * dt
        dR = dR @ dRk
    T = torch.full((K,), N * dt, dtype=torch.float64, device=DEV)
    m = dict(dR=dR, dv=dv, dp=dp, JRg=JRg, Jvg=Jvg, Jva=Jva, Jpg=Jpg, Jpa=Jpa, T=T, bg0=bg0, ba0=ba0)
    U = torch.linalg.cholesky(torch.linalg.inv(cov)).transpose(1, 2)       # inverse covariance = U^T U
    return m, U


class _Problem:
    """Edges as groups of (residual, whitened Jacobian) over the camera blocks (DB columns
    each) and the points."""

    def __init__(self, kind, p, fixed_first=False):
        self.vi = kind == "vi"
        self.DB = 15 if self.vi else 9
        self.cam = _dev(p.kf_idx if self.vi else p.cam_idx, torch.int64)
        self.pt = _dev(p.pt_idx, torch.int64)
        self.obs = _dev(p.obs)
        self.delta = p.huber_delta
        self.C, self.P = (p.n_kf if self.vi else p.n_cams), p.n_pts
        self.fixed = fixed_first
        if self.vi:
            c = p.camera
            self.rig = dict(fx=c["fx"], fy=c["fy"], cx=c["cx"], cy=c["cy"], b=c["baseline"], R=_dev(c["R_cb"]), t=_dev(c["t_cb"]))
            self.m, self.U = _preintegrate(p)
            self.rw = torch.cat([torch.full((3,), p.noise["sigma_bg"]), torch.full((3,), p.noise["sigma_ba"])]).to(DEV, torch.float64)
            self.prior = _dev(np.r_[np.full(3, 1e2), np.full(3, 1e1)])      # 1 / prior sigma

    def rot(self, cams):
        return _qrot(cams[:, :4]) if self.vi else _so3(cams[:, :3])

    def obs_args(self, cams, pts, s):
        c = self.cam[s]
        return cams[c], self.rot(cams)[c], pts[self.pt[s]], self.obs[s]

    def slices(self):
        n = self.cam.shape[0]
        return [slice(i, min(n, i + 1_000_000)) for i in range(0, n, 1_000_000)]

    def fn(self):
        if self.vi:
            return (lambda d, *a: _stereo_residual(d, *a, self.rig)), 9
        return _ba_residual, 12

    def imu(self, cams, want_J):
        """Camera-side rows: (first column block, second or -1, r, J [n, m, 30])."""
        if not self.vi:
            return []
        xi, xj, R = cams[:-1], cams[1:], self.rot(cams)
        z = torch.zeros(30, dtype=torch.float64, device=DEV)
        f = torch.func.vmap(_imu_residual, in_dims=(None, 0, 0, 0, 0, 0))
        a = (xi, xj, R[:-1], R[1:], self.m)
        i = torch.arange(self.C - 1, device=DEV)
        r = (self.U @ f(z, *a)[:, :, None])[:, :, 0]
        J = self.U @ torch.func.vmap(torch.func.jacfwd(_imu_residual), in_dims=(None, 0, 0, 0, 0, 0))(z, *a) if want_J else None
        s = 1.0 / (self.rw * torch.sqrt(self.m["T"])[:, None])
        rr = s * (xj[:, 10:16] - xi[:, 10:16])
        Jr = torch.zeros(self.C - 1, 6, 30, dtype=torch.float64, device=DEV)
        Jr[:, :, 9:15], Jr[:, :, 24:30] = -torch.diag_embed(s), torch.diag_embed(s)
        rp = (self.prior * cams[0, 10:16])[None]
        Jp = torch.zeros(1, 6, 30, dtype=torch.float64, device=DEV)
        Jp[0, :, 9:15] = torch.diag(self.prior)
        return [(i, i + 1, r, J), (i, i + 1, rr, Jr), (i[:1] * 0, i[:1] * 0, rp, Jp)]

    def cost(self, cams, pts):
        f, n = self.fn()
        z = torch.zeros(n, dtype=torch.float64, device=DEV)
        F = 0.0
        for s in self.slices():
            r = torch.func.vmap(f, in_dims=(None, 0, 0, 0, 0))(z, *self.obs_args(cams, pts, s))
            q = (r * r).sum(1)
            if self.delta is not None:
                q = torch.where(q > self.delta ** 2, 2 * self.delta * torch.sqrt(q) - self.delta ** 2, q)
            F += 0.5 * float(q.sum())
        return F + sum(0.5 * float((r * r).sum()) for _, _, r, _ in self.imu(cams, False))

    def rows(self, cams, pts):
        f, n = self.fn()
        z = torch.zeros(n, dtype=torch.float64, device=DEV)
        rs, Js = [], []
        for s in self.slices():
            a = self.obs_args(cams, pts, s)
            r = torch.func.vmap(f, in_dims=(None, 0, 0, 0, 0))(z, *a)
            J = torch.func.vmap(torch.func.jacfwd(f), in_dims=(None, 0, 0, 0, 0))(z, *a)
            if self.delta is not None:
                q = torch.sqrt((r * r).sum(1))
                w = torch.sqrt(torch.where(q > self.delta, self.delta / q, torch.ones_like(q)))
                r, J = r * w[:, None], J * w[:, None, None]
            rs.append(r)
            Js.append(J)
        r, J = torch.cat(rs), torch.cat(Js)
        Jc, Jp = J[:, :, :n - 3].contiguous(), J[:, :, n - 3:].contiguous()
        if self.fixed:
            Jc[self.cam == 0] = 0
        return r, Jc, Jp

    def retract(self, cams, dc):
        out = cams.clone()
        if self.vi:
            q = _qmul(cams[:, :4], _quat(dc[:, :3]))
            q = q / torch.linalg.vector_norm(q, dim=-1, keepdim=True)
            q = torch.where(q[:, 3:] < 0, -q, q)
            out[:, :4] = q
            out[:, 4:7] = cams[:, 4:7] + (self.rot(cams) @ dc[:, 3:6, None])[:, :, 0]
            out[:, 7:] = cams[:, 7:] + dc[:, 6:]
            return out
        q = _qmul(_quat(dc[:, :3]), _quat(cams[:, :3]))
        q = torch.where(q[:, 3:] < 0, -q, q)
        s = torch.linalg.vector_norm(q[:, :3], dim=-1, keepdim=True)
        out[:, :3] = q[:, :3] * torch.where(s < 1e-9, 2 * torch.ones_like(s), 2 * torch.atan2(s, q[:, 3:]) / s)
        out[:, 3:] = cams[:, 3:] + dc[:, 3:]
        return out if not self.fixed else torch.cat([cams[:1], out[1:]])


def _mv(J, x):
    return (J @ x[:, :, None])[:, :, 0]


def _solve(prob, cams, pts, lam, rows, ratio, full):
    """One damped step by PCG: (dc, dp, model decrease)."""
    r, Jc, Jp = rows
    C, P, DB, DC = prob.C, prob.P, prob.DB, Jc.shape[2]
    cam, pt = prob.cam, prob.pt
    z = lambda *s: torch.zeros(*s, dtype=torch.float64, device=DEV)  # noqa: E731
    add = lambda n, w, idx, v: z(n, *w).index_add_(0, idx, v)  # noqa: E731
    JcT, JpT = Jc.transpose(1, 2), Jp.transpose(1, 2)
    Hcc, bc = z(C, DB, DB), z(C, DB)
    Hcc[:, :DC, :DC] = add(C, (DC, DC), cam, JcT @ Jc)
    bc[:, :DC] = add(C, (DC,), cam, _mv(JcT, r))
    xs = prob.imu(cams, True)
    for i, j, rx, Jx in xs:
        Ji, Jj = Jx[:, :, :15], Jx[:, :, 15:]
        Hcc.index_add_(0, i, Ji.transpose(1, 2) @ Ji)
        bc.index_add_(0, i, _mv(Ji.transpose(1, 2), rx))
        Hcc.index_add_(0, j, Jj.transpose(1, 2) @ Jj)
        bc.index_add_(0, j, _mv(Jj.transpose(1, 2), rx))
    Hpp, bp = add(P, (3, 3), pt, JpT @ Jp), add(P, (3,), pt, _mv(JpT, r))
    D = lambda H: torch.diag_embed(torch.diagonal(H, dim1=1, dim2=2).clamp(1e-6, 1e32))  # noqa: E731
    Hc, Hp = Hcc + lam * D(Hcc), Hpp + lam * D(Hpp)
    Hi = torch.linalg.inv(Hp)

    def cams_H(x):      # (H_cc + lam D) x with the camera-side edges' coupling
        y = _mv(Hc, x)
        for i, j, _, Jx in xs:
            if i.shape[0] == 1 and C > 2:
                continue
            Ji, Jj = Jx[:, :, :15], Jx[:, :, 15:]
            y.index_add_(0, i, _mv(Ji.transpose(1, 2), _mv(Jj, x[j])))
            y.index_add_(0, j, _mv(Jj.transpose(1, 2), _mv(Ji, x[i])))
        return y

    def to_pt(x):       # H_pc x
        return add(P, (3,), pt, _mv(JpT, _mv(Jc, x[:, :DC][cam])))

    def to_cam(t):      # H_cp t
        y = z(C, DB)
        y[:, :DC] = add(C, (DC,), cam, _mv(JcT, _mv(Jp, t[pt])))
        return y

    if full:
        A = lambda v: (cams_H(v[0]) + to_cam(v[1]), _mv(Hp, v[1]) + to_pt(v[0]))  # noqa: E731
        Mc = torch.linalg.inv(Hc)
        M = lambda v: (_mv(Mc, v[0]), _mv(Hi, v[1]))  # noqa: E731
        g = (-bc, -bp)
    else:
        S = Hc.clone()
        W = JcT @ Jp
        S[:, :DC, :DC] -= add(C, (DC, DC), cam, W @ Hi[pt] @ W.transpose(1, 2))
        Mc = torch.linalg.inv(S)
        A = lambda v: (cams_H(v[0]) - to_cam(_mv(Hi, to_pt(v[0]))),)  # noqa: E731
        M = lambda v: (_mv(Mc, v[0]),)  # noqa: E731
        g = (-bc + to_cam(_mv(Hi, bp)),)
    dot = lambda a, b: sum(float((u * w).sum()) for u, w in zip(a, b))  # noqa: E731
    axpy = lambda s, a, b: tuple(s * u + w for u, w in zip(a, b))  # noqa: E731
    x, res = tuple(torch.zeros_like(u) for u in g), g
    zz = M(res)
    pdir, rz, gn = zz, dot(res, zz), math.sqrt(dot(g, g))
    best, rmin = x, gn
    for _ in range(100):
        y = A(pdir)
        pAp = dot(pdir, y)
        if not pAp > 0:
            break
        al = rz / pAp
        x, res = axpy(al, pdir, x), axpy(-al, y, res)
        n = math.sqrt(dot(res, res))
        if ratio > 0:
            if n < rmin:
                rmin, best = n, x
            elif n > ratio * rmin:
                x = best
                break
        zz = M(res)
        rz1 = dot(res, zz)
        if n <= 1e-6 * gn or not rz1 > 0:
            break
        pdir, rz = axpy(rz1 / rz, pdir, zz), rz1
    dc = x[0]
    dp = x[1] if full else _mv(Hi, -bp - to_pt(dc))
    Jd = _mv(Jc, dc[:, :DC][cam]) + _mv(Jp, dp[pt])
    L = -float((bc * dc).sum()) - float((bp * dp).sum()) - 0.5 * float((Jd * Jd).sum())
    for i, j, _, Jx in xs:
        v = _mv(Jx[:, :, :15], dc[i]) + _mv(Jx[:, :, 15:], dc[j])
        L -= 0.5 * float((v * v).sum())
    return dc, dp, L


def _lm(prob, cams, pts, iters, lam, ratio, full):
    F0 = F = prob.cost(cams, pts)
    nu, rows = 2.0, None
    for _ in range(iters):
        rows = rows or prob.rows(cams, pts)
        dc, dp, L = _solve(prob, cams, pts, lam, rows, ratio, full)
        c1, p1 = prob.retract(cams, dc), pts + dp
        F1 = prob.cost(c1, p1)
        if L > 0 and math.isfinite(F1) and F1 < F:
            rho = (F - F1) / L
            lam *= max(1.0 / 3.0, 1.0 - (2.0 * rho - 1.0) ** 3)
            cams, pts, F, nu, rows = c1, p1, F1, 2.0, None
        else:
            lam, nu = lam * nu, nu * 2.0
    return cams, pts, F0, F


def exact(case, seed):
    if case["kind"] == "cost":
        p = _scene(case, seed)
        return torch.tensor([_Problem("ba", p).cost(_dev(p.cams0), _dev(p.pts0))], dtype=torch.float64)
    full = case.get("solver") == "full"
    if case["kind"] == "vi":
        p = _vi(case, seed)
        todo = [(_Problem("vi", p), p.nav0, p.pts0)]
    elif case["kind"] == "batch":
        todo = [(_Problem("ba", p, True), p.cams0, p.pts0)
                for p in _windows(case, seed)]
    else:
        p = _scene(case, seed)
        todo = [(_Problem("ba", p, case["scene"] == "window"), p.cams0, p.pts0)]
    got = [_lm(q, _dev(c), _dev(x), case["iters"], case["damping"], 0.0 if case["kind"] == "vi" else 10.0, full)
           for q, c, x in todo]
    return dict(cams=torch.cat([g[0] for g in got]), pts=torch.cat([g[1] for g in got]),
                initial_cost=np.array([g[2] for g in got]), final_cost=np.array([g[3] for g in got]))
