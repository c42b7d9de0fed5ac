"""Single-frequency apply at the edges of its kernel (run with -m gpu): numbers of
right-hand sides per pass, conjugate points, near blocks wider than the column
tile, far blocks with more factor rows than a chunk, columns split over thread
groups.  Reference: the tensor's own rebuilt entries times x in FP64.  Tolerance
(relative 2-norm): rebuilt entries and products are sums of n <= 1280 terms in the
tensor's precision, error about sqrt(n) unit roundoffs of the sum of moduli, which
is within a factor 30 of the result for Gaussian x: 36 * 6e-8 * 30 = 6e-5 (mixed),
36 * 1.1e-16 * 30 = 1.2e-13 (FP64).
"""
import numpy as np
import pytest

from paper_2505_00715_gb300.inputs import icosphere, random_weights

pytestmark = pytest.mark.gpu
TOL = {"MIXED": 6e-5, "FP64": 1.2e-13}


@pytest.fixture(scope="module")
def td():
    import paper_2505_00715_gb300 as td
    return td


@pytest.fixture(scope="module")
def ctx(td):
    return td.Context(0)


@pytest.mark.parametrize("prec", ["MIXED", "FP64"])
@pytest.mark.parametrize("op,level,leaf,eps", [("SLP", 2, 7, 1e-4), ("DLP", 2, 16, 1e-6), ("SLP", 3, 700, 1e-4),
                                               ("SLP", 3, 160, 1e-7)])
def test_apply_one_sizes(td, ctx, op, level, leaf, eps, prec):
    import torch
    V, T = icosphere(level)
    gm = td.Mesh(ctx, V, T)
    f = td.Freqs.bdf2(ctx, 16, 0.1)
    nc = len(V) if op == "DLP" else len(T)
    tree = td.Tree(gm, td.P0, td.P1 if op == "DLP" else td.P0, leaf, 2.0)
    X = td.compress(gm, getattr(td, op), f, tree, eps=eps, eps_aca=eps / 100, prec=getattr(td, prec), balance=False)
    ct = torch.complex128 if prec == "FP64" else torch.complex64
    rows = np.arange(0, len(T), 1 if level == 2 else 37)
    for k in (0, 3, 13):
        rr, cc = np.meshgrid(rows, np.arange(nc), indexing="ij")
        A = X.entries(rr.ravel(), cc.ravel(), np.full(rr.size, k)).cpu().numpy().reshape(len(rows), nc).astype(complex)
        for nrhs in (1, 2, 3, 4, 6):
            x = random_weights(1, nc, nrhs, seed=k + nrhs)[0]
            xt = torch.as_tensor(x, dtype=ct, device="cuda")
            y = X.apply_freq(k, xt).cpu().numpy()[rows]
            ref = A @ xt.cpu().numpy().astype(complex)
            err = np.linalg.norm(y - ref) / np.linalg.norm(ref)
            assert err <= TOL[prec], (k, nrhs, err)
