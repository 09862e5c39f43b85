"""Solves whose bounded device waits give up (made to by gpo_debug_hold_waits: an arrival that
does not come; nothing faults and every kernel returns after about a second)."""
import numpy as np
import pytest

from paper_2509_26581_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpo():
    from paper_2509_26581_gb300 import gpo as m
    return m


# a solve by a cluster, by a whole grid, and in one launch on the matrix-free product
KINDS = {
    "cluster": (lambda: synth.ba_ring(2, 10, 500, 6), "fp64", 0),
    "grid": (lambda: synth.ba_path(4, 333, 20000, "geom"), "fp32", 0),
    "matrix_free": (lambda: synth.ba_path(3, 20, 2001, "pareto"), "bf16", 0),
}


def _build(gpo, kind, **kw):
    make, prec, variant = KINDS[kind]
    p = make()
    g, c0, p0 = gpo.ba_graph(p.cams0, p.pts0, p.cam_idx, p.pt_idx, p.obs, p.huber_delta, prec, spmv_variant=variant,
                             chunk_edges=512, **kw)
    return p, g, c0, p0


def _timeout(gpo, call):
    with pytest.raises(gpo.GpoError) as e:
        call()
    assert e.value.status == gpo.GPO_ERR_TIMEOUT


@pytest.mark.parametrize("kind", list(KINDS))
def test_a_wait_that_gives_up_is_reported(gpo, kind):
    _, g, _, _ = _build(gpo, kind)
    g.debug_hold_waits(True)
    _timeout(gpo, lambda: g.optimize(2))
    _timeout(gpo, lambda: gpo.optimize_batch([g, _build(gpo, kind)[1]], 2))


@pytest.mark.parametrize("kind", ["cluster", "matrix_free"])
def test_a_server_reports_a_wait_that_gives_up(gpo, kind):
    _, g, _, _ = _build(gpo, kind)
    g.debug_hold_waits(True)
    sv = gpo.Server(KINDS[kind][1])
    sv.submit(g, 2)
    _timeout(gpo, sv.step)
    sv.close()


def test_the_diagnostic_covers_a_clusters_wait(gpo):
    p, g, c0, _ = _build(gpo, "cluster")
    assert g.debug_wait_timeout() == gpo.GPO_ERR_TIMEOUT
    _, h, d0, _ = _build(gpo, "cluster")
    assert g.optimize(3).final_cost == h.optimize(3).final_cost
    assert np.array_equal(g.get_state(c0, p.n_cams, 9), h.get_state(d0, p.n_cams, 9))
