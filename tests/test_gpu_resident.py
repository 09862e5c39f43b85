"""The PCG of small mixed-precision systems in one launch (the automatic product where the
system's chunks fit the device at once) against the launches of the pipelined product
(variant 3).  The sums and their order are the same, so every comparison is bit for bit."""
import numpy as np
import pytest

from paper_2509_26581_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpo():
    from paper_2509_26581_gb300 import gpo as m
    return m


# one chunk; more camera units than chunks; up to 32 units and beyond; more than 32 camera
# blocks; ragged last chunk; two chunks per CTA
SCENES = {
    "one_chunk": lambda: synth.ba_ring(1, 2, 40, 2),
    "few_chunks": lambda: synth.ba_ring(2, 70, 300, 4, outlier_frac=0.02, huber_delta=2.0),
    "window": lambda: synth.ba_path(3, 20, 2001, "pareto"),
    "units_33": lambda: synth.ba_ring(4, 66, 4001, 5),
    "blocks_33": lambda: synth.ba_ring(5, 264, 3000, 6),
    "two_per_cta": lambda: synth.ba_path(6, 90, 60000, "geom"),
}


def _solve(gpo, p, variant, iters=3, chunk=0, **kw):
    g, cams, pts = gpo.ba_graph(p.cams0, p.pts0, p.cam_idx, p.pt_idx, p.obs, p.huber_delta, "bf16",
                                spmv_variant=variant, chunk_edges=chunk)
    r = g.optimize(iters, gpo.default_params(**kw))
    h = [(x["pcg_iters"], x["cost"], x["accepted"]) for x in g.history()]
    out = r.final_cost, r.final_lambda, r.pcg_iters_total, h, g.get_state(cams, p.n_cams, 9), g.get_state(pts, p.n_pts, 3)
    g.close()
    return out


def _same(a, b):
    assert a[:4] == b[:4]
    assert np.array_equal(a[4], b[4]) and np.array_equal(a[5], b[5])


@pytest.mark.parametrize("scene", list(SCENES))
def test_one_launch_solves_bit_for_bit_like_the_launches(gpo, scene):
    p = SCENES[scene]()
    _same(_solve(gpo, p, 0), _solve(gpo, p, 3))


# restarts, the rejection guard, no normalisation, the iteration cap, a heavy and a light damping
@pytest.mark.parametrize("kw", [dict(pcg_restart_every=4), dict(pcg_rejection_ratio=1.05), dict(pcg_normalize=0),
                                dict(pcg_max_iters=3), dict(initial_damping=10.0), dict(initial_damping=1e-8, pcg_tol=1e-9)],
                         ids=["restart", "reject", "plain", "cap", "heavy", "light"])
def test_stopping_rules(gpo, kw):
    p = synth.ba_path(7, 20, 2000, "pareto")
    _same(_solve(gpo, p, 0, **kw), _solve(gpo, p, 3, **kw))
    _same(_solve(gpo, p, 0, chunk=64, **kw), _solve(gpo, p, 3, chunk=64, **kw))


def test_batch_matches_the_graphs_alone(gpo):
    scenes = [synth.ba_path(20 + i, c, n, "pareto") for i, (c, n) in enumerate([(5, 300), (40, 8000), (17, 2500), (300, 900), (9, 11000)])]
    alone = [_solve(gpo, p, 3) for p in scenes]
    gs = [gpo.ba_graph(p.cams0, p.pts0, p.cam_idx, p.pt_idx, p.obs, p.huber_delta, "bf16", spmv_variant=0) for p in scenes]
    reps = gpo.optimize_batch([g for g, _, _ in gs], 3, gpo.default_params())
    for (g, cams, pts), r, a in zip(gs, reps, alone):
        assert (r.final_cost, r.final_lambda, r.pcg_iters_total) == a[:3]
        assert np.array_equal(g.get_state(cams, len(a[4]), 9), a[4])
        assert np.array_equal(g.get_state(pts, len(a[5]), 3), a[5])
        g.close()


def test_the_wait_is_bounded(gpo):
    p = synth.ba_path(3, 20, 2001, "pareto")
    g, _, _ = gpo.ba_graph(p.cams0, p.pts0, p.cam_idx, p.pt_idx, p.obs, None, "bf16")
    assert g.debug_wait_timeout() == gpo.GPO_ERR_TIMEOUT
    assert np.isfinite(g.optimize(2).final_cost)
    g.close()
