"""Weighted apply at the edges of its face kernel's tiles (run with -m gpu): right-hand
sides on both sides of the 16, 32 and 64 columns of a pass (odd ones with 8-byte
copies), one half only (all points real), face ranks and rows around the 16, 32 and
64-row tiles, blocks with more than 4 x 64 rows.  Reference: the tensor's own
single-frequency products summed in FP64 (another kernel).  Tolerance (relative
2-norm): split-BF16 contraction, about 1e-5 of the sum of moduli over the
frequencies; for Gaussian weights the sum of NQ terms' moduli is sqrt(NQ) = 4 times
its 2-norm: 4e-5.
"""
import numpy as np
import pytest

from paper_2505_00715_gb300.inputs import icosphere, random_weights

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def td():
    import paper_2505_00715_gb300 as td
    return td


@pytest.fixture(scope="module")
def ctx(td):
    return td.Context(0)


@pytest.mark.parametrize("op,level,leaf,real", [("SLP", 2, 12, False), ("DLP", 2, 16, False), ("SLP", 2, 33, True),
                                                ("SLP", 3, 330, False)])
def test_apply_faces_sizes(td, ctx, op, level, leaf, real):
    import torch
    V, T = icosphere(level)
    gm = td.Mesh(ctx, V, T)
    f = td.Freqs.points(ctx, np.linspace(0.5, 9.0, 7)) if real else td.Freqs.bdf2(ctx, 16, 0.1)
    nc = len(V) if op == "DLP" else len(T)
    tree = td.Tree(gm, td.P0, td.P1 if op == "DLP" else td.P0, leaf, 2.0)
    X = td.compress(gm, getattr(td, op), f, tree, eps=1e-6, eps_aca=1e-8, prec=td.MIXED, balance=False)
    for nrhs in (1, 3, 8, 9, 16, 17, 33, 40):
        W = torch.as_tensor(random_weights(f.NQ, nc, nrhs, seed=nrhs), dtype=torch.complex64, device="cuda")
        y = X.apply_weighted(W).to(torch.complex128)
        ref = sum(X.apply_freq(k, W[k].contiguous()).to(torch.complex128) for k in range(f.NQ))
        err = (torch.linalg.norm(y - ref) / torch.linalg.norm(ref)).item()
        assert err <= 4e-5, (nrhs, err)
