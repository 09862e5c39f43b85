"""True-residual restarts in the one-launch matrix-free PCG where there are more camera
units (two cameras each) than chunks, so that CTAs without chunks take part: a restart's
update must not overwrite the last residual norms while such a CTA still reads them.  Bit
for bit like the separate launches; a lost race gives other scalars or a wait that gives up."""
import numpy as np
import pytest

from paper_2509_26581_gb300 import synth

pytestmark = pytest.mark.gpu

# cameras, points, views -> chunks of 512 edges
SCENES = {"70_cams_3_chunks": (2, 70, 300, 4), "130_cams_1_chunk": (8, 130, 120, 4), "264_cams_18_chunks": (5, 264, 1500, 6)}


def _solve(p, variant, **kw):
    from paper_2509_26581_gb300 import gpo
    g, c0, p0 = gpo.ba_graph(p.cams0, p.pts0, p.cam_idx, p.pt_idx, p.obs, p.huber_delta, "bf16", spmv_variant=variant,
                             chunk_edges=512)
    r = g.optimize(3, gpo.default_params(pcg_rejection_ratio=0.0, pcg_tol=1e-12, pcg_max_iters=60, **kw))
    h = [(x["pcg_iters"], x["pcg_products"], x["cost"], x["accepted"]) for x in g.history()]
    info = g.info()
    out = r.final_cost, r.final_lambda, h, g.get_state(c0, p.n_cams, 9), g.get_state(p0, p.n_pts, 3)
    g.close()
    return out, info


@pytest.mark.parametrize("every", [4, 5, 9])
@pytest.mark.parametrize("scene", list(SCENES))
def test_restarts_with_units_without_chunks(scene, every):
    p = synth.ba_ring(*SCENES[scene], outlier_frac=0.02, huber_delta=2.0)
    want, info = _solve(p, 3, pcg_restart_every=every)
    assert info["chunks"] < 4 * ((p.n_cams + 7) // 8)
    assert any(products > its for its, products, _, _ in want[2])      # restarts took place
    for _ in range(5):
        got, _ = _solve(p, 0, pcg_restart_every=every)
        assert got[:3] == want[:3]
        assert np.array_equal(got[3], want[3]) and np.array_equal(got[4], want[4])
