"""Graphs that are finalized inside a call that solves them on another graph's or a server's
stream: their uploads (and the row-pair plans of the explicit Schur complement, kernels on
the graph's own stream) come first, so the results are those of the graphs alone, bit for
bit.  The largest plan comes last: nothing between its upload and the solve gives it time."""
import numpy as np
import pytest

from paper_2509_26581_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpo():
    from paper_2509_26581_gb300 import gpo as m
    return m


@pytest.fixture(scope="module")
def scenes():
    return [synth.ba_ring(1, 10, 500, 6), synth.ba_path(2, 40, 9000, "pareto"), synth.ba_path(3, 300, 60000, "geom")]


def _build(gpo, p, prec, **kw):
    return gpo.ba_graph(p.cams0, p.pts0, p.cam_idx, p.pt_idx, p.obs, p.huber_delta, prec, spmv_variant=0,
                        chunk_edges=512, **kw)


def _result(p, built, rep):
    g, c0, p0 = built
    return rep.final_cost, rep.pcg_iters_total, g.get_state(c0, p.n_cams, 9), g.get_state(p0, p.n_pts, 3)


def _same(a, b):
    assert a[:2] == b[:2] and np.array_equal(a[2], b[2]) and np.array_equal(a[3], b[3])


@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16"])
def test_batch_of_fresh_graphs_waits_for_their_uploads(gpo, scenes, prec):
    alone = []
    for p in scenes:
        b = _build(gpo, p, prec)
        alone.append(_result(p, b, b[0].optimize(2)))
    for _ in range(3):
        built = [_build(gpo, p, prec) for p in scenes]
        for b in built:
            b[0].plan()   # host part first: the uploads follow one another and the solve at once
        reps = gpo.optimize_batch([b[0] for b in built], 2)
        for p, b, r, a in zip(scenes, built, reps, alone):
            _same(_result(p, b, r), a)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_server_waits_for_the_uploads_of_graphs_with_their_own_streams(gpo, scenes, prec):
    import torch
    streams = [torch.cuda.Stream() for _ in scenes]
    alone = []
    for p in scenes:
        b = _build(gpo, p, prec)
        alone.append(_result(p, b, b[0].optimize(3)))
    sv = gpo.Server(prec)
    built = [_build(gpo, p, prec, stream=s.cuda_stream) for p, s in zip(scenes, streams)]
    tickets = [sv.submit(b[0], 3) for b in built]
    while sum(sv.step()[:2]):
        pass
    for p, b, t, a in zip(scenes, built, tickets, alone):
        _same(_result(p, b, sv.poll(t)), a)
    sv.close()
