"""Graphs on a caller's allocator, and memory that holds a graph only without the explicit
Schur complement: what finalizing writes, that nothing relies on what the memory held before,
and that such a graph is solved matrix-free rather than refused."""
import ctypes

import numpy as np
import pytest

from paper_2509_26581_gb300 import synth

pytestmark = pytest.mark.gpu

FILL = 0x5A


@pytest.fixture(scope="module")
def gpo():
    from paper_2509_26581_gb300 import gpo as m
    return m


class Arenas:
    """Allocator hooks over torch tensors filled with one byte; refuses more than `limit`."""

    def __init__(self, gpo, limit=None):
        import torch
        self.blocks, self.asked = {}, []

        def alloc(n, ctx):
            self.asked.append(n)
            if limit is not None and n > limit:
                return 0
            t = torch.full((n + 256,), FILL, dtype=torch.uint8, device="cuda")
            torch.cuda.synchronize()
            p = (t.data_ptr() + 255) // 256 * 256
            self.blocks[p] = t[p - t.data_ptr():][:n]
            return p

        self.alloc = gpo._ALLOC(alloc)
        self.free = gpo._FREE(lambda p, ctx: self.blocks.pop(p, None) is None and None)

    def graph(self, gpo, p, prec, variant=0):
        """gpo.ba_graph on this allocator."""
        d = gpo.gpo_graph_desc()
        gpo._check(gpo.lib.gpo_graph_desc_default(ctypes.byref(d)))
        d.precision, d.chunk_edges, d.spmv_variant = gpo.PRECISIONS[prec], 512, variant
        d.alloc, d.free = self.alloc, self.free
        g = gpo.Graph.__new__(gpo.Graph)
        g.h, g.precision = ctypes.c_void_p(), prec
        gpo._check(gpo.lib.gpo_graph_create(ctypes.byref(d), ctypes.byref(g.h)))
        c0 = g.add_vertices(gpo.GPO_V_BA_CAMERA9, 9, p.n_cams)
        p0 = g.add_vertices(gpo.GPO_V_POINT3, 3, p.n_pts)
        g.add_edges(gpo.GPO_E_BA_REPROJ, np.stack([p.cam_idx + c0, p.pt_idx + p0], 1).astype(np.int64), p.obs, None,
                    gpo.GPO_LOSS_HUBER, float(p.huber_delta))
        g.set_initial(c0, p.cams0)
        g.set_initial(p0, p.pts0)
        return g, c0, p0


@pytest.mark.parametrize("prec,kernel", [("fp64", 7), ("fp32", 7), ("bf16", 3)])
def test_only_the_uploaded_arrays_are_written(gpo, prec, kernel):
    """After finalizing, arrays that only solves write still hold the allocator's bytes: they
    (partial sums, blocks, camera rows, point blocks) are more than a quarter of the arena.
    A graph in such memory solves bit for bit like one in fresh memory."""
    p = synth.ba_path(1, 200, 30_000, "pareto")
    arenas = Arenas(gpo)
    g, c0, p0 = arenas.graph(gpo, p, prec)
    g.optimize(0)
    block, = arenas.blocks.values()
    assert g.info()["spmv_kernel"] == kernel and block.numel() == g.footprint()
    assert int((block == FILL).sum()) > block.numel() / 4
    h, d0, q0 = gpo.ba_graph(p.cams0, p.pts0, p.cam_idx, p.pt_idx, p.obs, p.huber_delta, prec, spmv_variant=0,
                             chunk_edges=512)
    a, b = (x.optimize(3, gpo.default_params(initial_damping=0.1)) for x in (g, h))
    assert (a.final_cost, a.pcg_iters_total, a.accepted) == (b.final_cost, b.pcg_iters_total, b.accepted)
    assert np.array_equal(g.get_state(c0, p.n_cams, 9), h.get_state(d0, p.n_cams, 9))
    assert np.array_equal(g.get_state(p0, p.n_pts, 3), h.get_state(q0, p.n_pts, 3))
    g.close()
    assert not arenas.blocks


def _sizes(gpo, p, prec):
    """Planned bytes with the explicit Schur complement, and where a budget leaves it out."""
    out = []
    for budget in (0, -1):
        g = gpo.ba_graph(p.cams0, p.pts0, p.cam_idx, p.pt_idx, p.obs, p.huber_delta, prec, spmv_variant=0,
                         chunk_edges=512, memory_budget=out[0] + budget if budget else 0)[0]
        out.append(g.plan())
        g.close()
    assert out[0] > 1.1 * out[1]
    return out


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_an_allocator_that_holds_the_graph_only_without_the_blocks(gpo, prec):
    p = synth.ba_path(3, 121, 9000, "pareto")
    full, plain = _sizes(gpo, p, prec)
    arenas = Arenas(gpo, limit=(full + plain) // 2)
    g, c0, _ = arenas.graph(gpo, p, prec)
    rep = g.optimize(2)
    assert arenas.asked == [full, plain] and g.footprint() == plain and g.info()["spmv_kernel"] != 7
    h, d0, _ = gpo.ba_graph(p.cams0, p.pts0, p.cam_idx, p.pt_idx, p.obs, p.huber_delta, prec, spmv_variant=0,
                            chunk_edges=512, memory_budget=(full + plain) // 2)
    assert rep.final_cost == h.optimize(2).final_cost
    assert np.array_equal(g.get_state(c0, p.n_cams, 9), h.get_state(d0, p.n_cams, 9))
    none = Arenas(gpo, limit=plain - 1)
    with pytest.raises(gpo.GpoError) as e:
        none.graph(gpo, p, prec)[0].optimize(1)
    assert e.value.status == gpo.GPO_ERR_OOM and none.asked == [full, plain]


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_a_server_budget_that_holds_the_graph_only_without_the_blocks(gpo, prec):
    p = synth.ba_path(3, 121, 9000, "pareto")
    full, plain = _sizes(gpo, p, prec)

    def graph(**kw):
        return gpo.ba_graph(p.cams0, p.pts0, p.cam_idx, p.pt_idx, p.obs, p.huber_delta, prec, spmv_variant=0,
                            chunk_edges=512, **kw)

    h, d0, _ = graph(memory_budget=plain)
    ref = h.optimize(2)
    g, c0, _ = graph()
    sv = gpo.Server(prec, memory_budget=plain)
    ticket = sv.submit(g, 2)
    while sum(sv.step()[:2]):
        assert sv.memory() == plain
    rep = sv.poll(ticket)
    assert (rep.final_cost, rep.pcg_iters_total) == (ref.final_cost, ref.pcg_iters_total)
    assert np.array_equal(g.get_state(c0, p.n_cams, 9), h.get_state(d0, p.n_cams, 9))
    with pytest.raises(gpo.GpoError) as e:
        gpo.Server(prec, memory_budget=plain - 1).submit(graph()[0], 2)
    assert e.value.status == gpo.GPO_ERR_OOM
    sv.close()
