"""Far-field fibres at the edges of their lane groups (run with -m gpu): blocks of one
row or column, fewer columns than a warp's four groups, sizes around a multiple of
the CTA's 16 groups, P1 columns, both forms, with and without dense working faces.
Reference: tdbem_entries.  Tolerance: the compression's eps per block gives
||C - C_r||_F <= 3 eps ||C||_F over the tensor (as tests/test_gpu_parity.py).
"""
import numpy as np
import pytest

from paper_2505_00715_gb300.inputs import icosphere

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["MIXED", "FP64"])
@pytest.mark.parametrize("op", ["SLP", "DLP", "ADLP"])
@pytest.mark.parametrize("leaf,dense", [(1, True), (3, True), (3, False), (13, True), (17, True)])
def test_far_fibre_sizes(leaf, dense, op, prec):
    import paper_2505_00715_gb300 as td
    ctx = td.Context(0)
    V, T = icosphere(2)
    V = V * np.array([1.0, 1.3, 2.1])  # no two triangles alike
    gm = td.Mesh(ctx, V, T)
    f = td.Freqs.bdf2(ctx, 6, 0.2)
    nc = len(V) if op == "DLP" else len(T)
    tree = td.Tree(gm, td.P0, td.P1 if op == "DLP" else td.P0, leaf, 2.0)
    eps = 1e-4
    X = td.compress(gm, getattr(td, op), f, tree, eps=eps, eps_aca=1e-6, prec=getattr(td, prec), dense_faces=dense)
    assert X.stats()["nfar"] > 0
    rr, cc = np.meshgrid(np.arange(len(T)), np.arange(nc), indexing="ij")
    num = den = 0.0
    for k in f.unique:
        reb = X.entries(rr.ravel(), cc.ravel(), np.full(rr.size, k)).cpu().numpy().reshape(len(T), nc)
        ref = td.entries(gm, getattr(td, op), f, np.arange(len(T)), np.arange(nc), [k], prec=td.FP64).cpu().numpy()[0]
        num += np.linalg.norm(reb - ref) ** 2
        den += np.linalg.norm(ref) ** 2
    assert np.sqrt(num / den) < 3 * eps
