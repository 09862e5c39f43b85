"""Planning of the explicit Schur complement from observations in any order: the tables of
cameras that share points come out the same, and a camera that sees a point twice is found
wherever its observations stand.  Tolerance: FP64 steps of three PCG iterations differ by
rounding (1e-10 of the largest entry, as for the product's other orders of summation)."""
import numpy as np
import pytest

from paper_2509_26581_gb300 import synth

pytestmark = pytest.mark.gpu


def _order(p, name):
    n = len(p.cam_idx)
    return {"camera": np.lexsort((p.pt_idx, p.cam_idx)), "point": np.lexsort((p.cam_idx, p.pt_idx)),
            "reversed": np.lexsort((p.cam_idx, p.pt_idx))[::-1], "shuffled": np.random.default_rng(1).permutation(n)}[name]


def _graph(p, i, variant):
    from paper_2509_26581_gb300 import gpo
    return gpo.ba_graph(p.cams0, p.pts0, p.cam_idx[i], p.pt_idx[i], p.obs[i], p.huber_delta, "fp64", spmv_variant=variant,
                        chunk_edges=512)[0]


@pytest.mark.parametrize("order", ["camera", "point", "reversed", "shuffled"])
@pytest.mark.parametrize("scene", [lambda: synth.ba_ring(3, 70, 900, 5), lambda: synth.ba_path(4, 200, 9000, "geom")],
                         ids=["ring", "path"])
def test_any_order_of_the_observations(scene, order):
    from paper_2509_26581_gb300 import gpo
    p = scene()
    i = _order(p, order)
    steps = []
    for variant in (2, 0):
        g = _graph(p, i, variant)
        dx, its = g.debug_step(1e-2, 9 * p.n_cams + 3 * p.n_pts, gpo.default_params(pcg_max_iters=3, pcg_tol=0.0))
        assert its == 3 and g.info()["spmv_kernel"] == (7 if variant == 0 else 2)
        steps.append(dx)
        g.close()
    assert np.max(np.abs(steps[1] - steps[0])) <= 1e-10 * np.max(np.abs(steps[0]))


@pytest.mark.parametrize("order", ["camera", "point", "reversed", "shuffled"])
def test_a_camera_that_sees_a_point_twice(order):
    p = synth.ba_ring(3, 70, 900, 5)
    i = _order(p, order)
    twice = np.r_[i, i[len(i) // 2]]      # first and last of the point's observations, or between others
    g = _graph(p, twice, 0)
    g.optimize(1)
    assert g.info()["spmv_kernel"] == 2 and np.isfinite(g.cost())
    g.close()
