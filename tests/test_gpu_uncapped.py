"""pcg_max_iters at the largest values of its type: solves end at their tolerance, as under any
cap they do not reach."""
import numpy as np
import pytest

from paper_2509_26581_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cap", [2**31 - 1, 2**31 - 2, 1717986917, 1717986918])
@pytest.mark.parametrize("prec,variant,solver", [("bf16", 0, 0), ("bf16", 3, 0), ("fp64", 0, 0), ("fp64", 2, 0), ("fp32", 0, 1)])
def test_a_cap_that_is_not_reached(prec, variant, solver, cap):
    from paper_2509_26581_gb300 import gpo
    p = synth.ba_path(3, 20, 2001, "pareto")
    out = []
    for n in (1000, cap):
        g, c0, p0 = gpo.ba_graph(p.cams0, p.pts0, p.cam_idx, p.pt_idx, p.obs, p.huber_delta, prec, spmv_variant=variant,
                                 chunk_edges=512)
        r = g.optimize(2, gpo.default_params(initial_damping=0.1, pcg_max_iters=n,
                                             solver=gpo.GPO_SOLVER_FULL if solver else 0))
        out.append((r.final_cost, r.pcg_iters_total, g.get_state(c0, p.n_cams, 9), g.get_state(p0, p.n_pts, 3)))
        g.close()
    assert out[0][:2] == out[1][:2] and 0 < out[0][1] < 1000
    assert np.array_equal(out[0][2], out[1][2]) and np.array_equal(out[0][3], out[1][3])
