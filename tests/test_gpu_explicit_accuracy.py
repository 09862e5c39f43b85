"""Diagonal blocks of the explicit Schur complement in FP32 where cameras see very many points:
against FP64 they are as exact as the matrix-free kernels' blocks of the same graph (a memory
budget leaves the explicit arrays out; points, chunks and so H_cc are the same to the bit).
Errors relative to the entries' diagonals, RMS over a scene, in units of 2^-23.  Both subtract
one sum of squares from the same H_cc; with sums in short chains each rounds like a few
additions, whatever the number of rows, so the two errors differ by their rows' own roundings:
15 % are allowed."""
import numpy as np
import pytest

from paper_2509_26581_gb300 import synth

pytestmark = pytest.mark.gpu


def _schur(p, prec, variant, kernel, **kw):
    from paper_2509_26581_gb300 import gpo
    g = gpo.ba_graph(p.cams0, p.pts0, p.cam_idx, p.pt_idx, p.obs, p.huber_delta, prec, spmv_variant=variant,
                     chunk_edges=512, **kw)[0]
    full = g.plan()
    S, _ = g.debug_schur(1e-2, p.n_cams)
    assert g.info()["spmv_kernel"] == kernel
    g.close()
    return S, full


# rows per camera: 33,000, 45,000, 20,000
@pytest.mark.parametrize("scene", [(21, 6, 50_000, 4), (22, 4, 60_000, 3), (23, 12, 40_000, 6)])
def test_fp32_sums_over_many_rows(scene):
    p = synth.ba_ring(*scene)
    exact, _ = _schur(p, "fp64", 2, 2)
    explicit, full = _schur(p, "fp32", 0, 7)
    free, _ = _schur(p, "fp32", 0, 3, memory_budget=full - 1)
    d = np.sqrt(np.einsum("cii->ci", exact))
    e, f = (float(np.sqrt((((S - exact) / (d[:, :, None] * d[:, None, :])) ** 2).mean())) * 2**23 for S in (explicit, free))
    assert e <= 1.15 * f, (e, f)
