"""The cost kernels (camera blocks formed once per run of one camera; reciprocal and square
root by iterations) against the same cost in extended precision.

Tolerance: an edge's projection rounds within about 32 eps of its size and the measurement's,
so its rho within 32 eps * 2 |r| (|u| + |z|) and the sum within the sum of these."""
import ctypes

import numpy as np
import pytest

from paper_2509_26581_gb300 import synth

pytestmark = pytest.mark.gpu


def _cost(cams, pts, ci, pi, obs, delta):
    """Cost and its tolerance, extended precision."""
    c, X, z = (np.asarray(a, dtype=np.longdouble) for a in (cams[ci], pts[pi], obs))
    w = c[:, :3]
    t = np.sqrt((w * w).sum(1))[:, None]
    t = np.where(t == 0, np.longdouble(1e-300), t)
    k = w / t
    P = (X * np.cos(t) + np.cross(k, X) * np.sin(t) + k * (k * X).sum(1)[:, None] * (1 - np.cos(t))) + c[:, 3:6]
    p = -P[:, :2] / P[:, 2:]
    r2 = (p * p).sum(1)
    u = (c[:, 6] * (1 + c[:, 7] * r2 + c[:, 8] * r2 * r2))[:, None] * p
    r = u - z
    s = (r * r).sum(1)
    rho = np.where((s > delta * delta) & (delta > 0), 2 * delta * np.sqrt(s) - delta * delta, s)
    eps = np.finfo(np.float64).eps
    tol = 32 * eps * (2 * np.sqrt(s) * (np.linalg.norm(u.astype(float), axis=1) + np.linalg.norm(z.astype(float), axis=1))).sum()
    return float(rho.sum() / 2), float(tol + 4 * eps * rho.sum())


def _noalloc(gpo, cams, pts, ci, pi, obs, delta):
    import torch
    dev = [torch.from_numpy(np.ascontiguousarray(a, dtype=t)).cuda()
           for a, t in ((cams, "f8"), (pts, "f8"), (ci, "i4"), (pi, "i4"), (obs, "f8"))]
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    st = gpo.lib.gpo_ba_cost_noalloc(0, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream),
                                     *[ctypes.c_void_p(t.data_ptr()) for t in dev], len(ci), delta,
                                     ctypes.c_void_p(out.data_ptr()))
    assert st == gpo.GPO_OK
    return float(out.item())


# around a warp, a CTA (256 edges) and two; cameras in runs, in no order, and alternating
@pytest.mark.parametrize("order", ["runs", "shuffled", "alternating"])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 255, 256, 257, 513, 3000])
def test_cost_matches_extended_precision(n, order):
    from paper_2509_26581_gb300 import gpo
    p = synth.ba_ring(5, 12, 800, 5, outlier_frac=0.05, huber_delta=1.0)
    idx = {"runs": lambda: np.argsort(p.cam_idx, kind="stable"),
           "shuffled": lambda: np.random.default_rng(n).permutation(len(p.cam_idx)),
           "alternating": lambda: np.arange(len(p.cam_idx))}[order]()[:n]
    for delta in (-1.0, 1.0):
        args = p.cams0, p.pts0, p.cam_idx[idx], p.pt_idx[idx], p.obs[idx]
        want, tol = _cost(*args, delta)
        assert abs(_noalloc(gpo, *args, delta) - want) <= tol
        g, _, _ = gpo.ba_graph(*args, delta if delta > 0 else None, "fp64")
        assert abs(g.cost() - want) <= tol
        g.close()


# zero depth, infinite depth, an infinite measurement, depths whose reciprocal is beyond the
# iteration's range, and a threshold whose square is subnormal: as plain arithmetic has them
@pytest.mark.parametrize("case", ["zero", "inf_depth", "inf_obs", "nan", "tiny", "huge", "tiny_delta"])
def test_cost_at_the_ends_of_the_range(case):
    from paper_2509_26581_gb300 import gpo
    cams = np.array([[0, 0, 0, 0, 0, 0, 1.0, 0, 0]])
    pts, obs, delta = np.array([[3.0, 4.0, -1.0]]), np.array([[1.0, 2.0]]), -1.0
    if case == "zero":
        pts[0, 2] = 0.0
    elif case == "inf_depth":
        cams[0, 5] = np.inf
    elif case == "inf_obs":
        obs[0, 0], delta = np.inf, 2.0
    elif case == "nan":
        obs[0, 0], delta = np.nan, 2.0
    elif case == "tiny":
        pts[0] = (3e-305, 4e-305, -1e-305)
    elif case == "huge":
        pts[0] = (3e305, 4e305, -1e305)
    elif case == "tiny_delta":
        pts[0], obs[0], delta = (0.0, 3e-160, -1.0), (0.0, 0.0), 1e-160
    z = np.zeros(1, np.int64)
    p = -pts[0, :2] / (pts[0, 2] + cams[0, 5]) if case != "zero" else np.array([np.inf, np.inf])
    with np.errstate(invalid="ignore"):
        p = p * (1 + 0.0 * (p * p).sum())       # distortion by zero coefficients: infinity gives NaN
        s = float(((p - obs[0]) ** 2).sum())
    want = 0.5 * (2 * delta * np.sqrt(s) - delta * delta if delta > 0 and s > delta * delta else s)
    got = _noalloc(gpo, cams, pts, z, z, obs, delta)
    if np.isfinite(want):
        assert abs(got - want) <= 1e-14 * abs(want) + 1e-323
    else:
        assert np.isnan(got) == np.isnan(want) and np.isinf(got) == np.isinf(want)
