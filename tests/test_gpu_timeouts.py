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
    g.debug_hold_waits(1)
    _timeout(gpo, lambda: g.optimize(2))
    _timeout(gpo, lambda: gpo.optimize_batch([g, _build(gpo, kind)[1]], 2))


@pytest.mark.parametrize("kind", ["cluster", "matrix_free"])
def test_a_server_reports_a_wait_that_gives_up(gpo, kind):
    _, g, _, _ = _build(gpo, kind)
    g.debug_hold_waits(1)
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


def _damped(gpo):
    """A damping at which the path scenes accept their first steps."""
    return gpo.default_params(initial_damping=0.1)


@pytest.mark.parametrize("kind", list(KINDS))
def test_a_lost_solve_takes_no_step_and_leaves_no_stale_cost(gpo, kind):
    """Two iterations, then one whose solve is lost: the graph is where a graph of two
    iterations is, says so, and goes on from there."""
    p, g, c0, p0 = _build(gpo, kind)
    _, h, d0, q0 = _build(gpo, kind)
    start = g.cost()
    two = h.optimize(2, _damped(gpo))
    assert two.accepted == 2
    g.debug_hold_waits(3)
    _timeout(gpo, lambda: g.optimize(4, _damped(gpo)))
    g.debug_hold_waits(0)

    def same():
        assert np.array_equal(g.get_state(c0, p.n_cams, 9), h.get_state(d0, p.n_cams, 9))
        assert np.array_equal(g.get_state(p0, p.n_pts, 3), h.get_state(q0, p.n_pts, 3))

    same()
    assert g.cost() == two.final_cost != start
    a, b = g.optimize(2, _damped(gpo)), h.optimize(2, _damped(gpo))
    assert (a.initial_cost, a.final_cost, a.pcg_iters_total) == (b.initial_cost, b.final_cost, b.pcg_iters_total)
    same()


@pytest.mark.parametrize("kind", list(KINDS))
def test_a_lost_solve_in_a_batch(gpo, kind):
    p, g, c0, _ = _build(gpo, kind)
    _, h, d0, _ = _build(gpo, kind)
    two = h.optimize(2, _damped(gpo))
    other = _build(gpo, kind)[1]
    g.debug_hold_waits(3)
    _timeout(gpo, lambda: gpo.optimize_batch([other, g], 3, _damped(gpo)))
    for x in (g, other):
        assert x.cost() == two.final_cost
        assert np.array_equal(x.get_state(c0, p.n_cams, 9), h.get_state(d0, p.n_cams, 9))


@pytest.mark.parametrize("kind", ["cluster", "matrix_free"])
def test_a_server_makes_a_lost_iteration_again(gpo, kind):
    p, g, c0, _ = _build(gpo, kind)
    _, h, d0, _ = _build(gpo, kind)
    ref = h.optimize(3, _damped(gpo))
    g.debug_hold_waits(2)
    sv = gpo.Server(KINDS[kind][1])
    ticket = sv.submit(g, 3, _damped(gpo))
    assert sv.step()[0] == 1
    _timeout(gpo, sv.step)
    g.debug_hold_waits(0)
    assert sv.step()[0] == 1 and sv.poll(ticket) is None
    assert sv.step() == (0, 0, 1)
    rep = sv.poll(ticket)
    assert (rep.final_cost, rep.iterations, rep.pcg_iters_total) == (ref.final_cost, 3, ref.pcg_iters_total)
    assert np.array_equal(g.get_state(c0, p.n_cams, 9), h.get_state(d0, p.n_cams, 9))
    sv.close()
