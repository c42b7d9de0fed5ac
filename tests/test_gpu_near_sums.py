"""Near-field sums at the edges of their kernels' ranges (run with -m gpu): the
FP64 separated frequency sums (number of frequencies, |s| from the shortest to
beyond the longest Chebyshev variant, Gauss orders, columns with more touching
triangles than an entry keeps) and tdbem_entries (few and many entries, with and
without the separated touching sums, invalid indices) against the FP64 oracle, and
the mixed form's on-demand near entries against the near-field tensor kernel.

Tolerances: 1e-12 (FP64) and 1e-5 (mixed) of an entry's sum of moduli, as the entry paths are
held to (tests/test_gpu_entry_paths.py).  On-demand entries: the approximation
of a near block interpolates the first selected frequency's slice, up to the FP32
rounding of at most 33 later terms of size <= the slice maximum: 33 * 2^-23 * 4
< 2e-5 of that maximum.
"""
import numpy as np
import pytest

from paper_2505_00715_gb300.inputs import icosphere

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def td():
    import paper_2505_00715_gb300 as td
    return td


@pytest.fixture(scope="module")
def ctx(td):
    return td.Context(0)


def _fan(n):
    """Double cone over an n-gon: two vertices of valence n."""
    a = 2 * np.pi * np.arange(n) / n
    V = np.vstack([np.c_[np.cos(a), np.sin(a), 0.03 * np.cos(3 * a)], [[0, 0, 0.6], [0, 0, -0.7]]])
    T = [(k, (k + 1) % n, n) for k in range(n)] + [((k + 1) % n, k, n + 1) for k in range(n)]
    return V, np.array(T, dtype=np.int32)


@pytest.mark.parametrize("op", ["SLP", "DLP", "ADLP"])
@pytest.mark.parametrize("mesh,scale,nf,ng", [("sphere", 1.0, 1, 5), ("sphere", 1.0, 2, 5), ("sphere", 0.05, 5, 3),
                                              ("sphere", 6.0, 9, 2), ("sphere", 40.0, 7, 5), ("fan", 2.0, 3, 1),
                                              ("fan", 1.0, 4, 7)])
def test_separated_sums(td, ctx, orc, op, mesh, scale, nf, ng):
    V, T = icosphere(1) if mesh == "sphere" else _fan(17)
    gm, om = td.Mesh(ctx, V, T), orc.Mesh(V, T)
    s = scale * np.array([0.3 + 0.1j * k + 0.35 * k for k in range(nf)])
    f = td.Freqs.points(ctx, s)
    rows = np.arange(0, len(T), 3, dtype=np.int32)
    cols = np.arange(len(V) if op == "DLP" else len(T), dtype=np.int32)
    fidx = np.arange(nf, dtype=np.int32)
    g = td.entries(gm, getattr(td, op), f, rows, cols, fidx, prec=td.FP64, ng=ng, path=td.PATH_NEAR).cpu().numpy()
    o = om.entries(getattr(orc, op), rows, cols, s, ng=ng)
    mag = om.entries_mag(getattr(orc, op), rows, cols, s, ng=ng)
    scale_k = mag.reshape(nf, -1).max(axis=1)
    err = np.abs(g - o) / np.maximum(mag, 1e-6 * scale_k[:, None, None])
    assert err.max() <= 1e-12, err.max()


@pytest.mark.parametrize("op", ["SLP", "DLP", "ADLP"])
@pytest.mark.parametrize("mesh", ["sphere", "fan"])
def test_on_demand_entries(td, ctx, op, mesh):
    """One near block over the whole mesh (a leaf as large as the mesh)."""
    V, T = icosphere(2) if mesh == "sphere" else _fan(31)
    gm = td.Mesh(ctx, V, T)
    f = td.Freqs.bdf2(ctx, 64, 0.4)
    nc = len(V) if op == "DLP" else len(T)
    tree = td.Tree(gm, td.P0, td.P1 if op == "DLP" else td.P0, 400, 2.0)
    X = td.compress(gm, getattr(td, op), f, tree, eps=1e-4, prec=td.MIXED)
    assert X.stats()["nnear"] == X.stats()["nblocks"] == 1
    k = int(f.unique[X.blocks()[2][0, 0]])
    rr, cc = np.meshgrid(np.arange(len(T)), np.arange(nc), indexing="ij")
    reb = X.entries(rr.ravel(), cc.ravel(), np.full(rr.size, k)).cpu().numpy().reshape(len(T), nc)
    ref = td.entries(gm, getattr(td, op), f, np.arange(len(T)), np.arange(nc), [k], prec=td.MIXED,
                     path=td.PATH_NEAR).cpu().numpy()[0]
    assert np.abs(reb - ref).max() <= 2e-5 * np.abs(ref).max()


@pytest.mark.parametrize("prec,tol", [("FP64", 1e-12), ("MIXED", 1e-5)])
@pytest.mark.parametrize("op", ["SLP", "DLP", "ADLP"])
@pytest.mark.parametrize("nr,nf,scale", [(1, 1, 1.0), (3, 7, 1.0), (34, 1, 1.0), (34, 2, 1.0), (34, 3, 1.0),
                                         (34, 6, 8.0), (34, 6, 60.0)])
def test_entries_sizes(td, ctx, orc, op, prec, tol, nr, nf, scale):
    V, T = _fan(17)
    gm, om = td.Mesh(ctx, V, T), orc.Mesh(V, T)
    s = scale * np.array([0.4 + 0.2j * k for k in range(nf + 1)])
    f = td.Freqs.points(ctx, s)
    ncol = len(V) if op == "DLP" else len(T)
    rows = np.arange(nr, dtype=np.int32)
    cols = np.tile(np.arange(ncol, dtype=np.int32), 1 + 520 // ncol) if nr > 3 else np.arange(0, ncol, 2, dtype=np.int32)
    fidx = np.arange(nf, 0, -1, dtype=np.int32)
    g = td.entries(gm, getattr(td, op), f, rows, cols, fidx, prec=getattr(td, prec)).cpu().numpy()
    o = om.entries(getattr(orc, op), rows, cols, s[fidx], ng=5)
    mag = om.entries_mag(getattr(orc, op), rows, cols, s[fidx], ng=5)
    err = np.abs(g - o) / np.maximum(mag, 1e-6 * mag.reshape(nf, -1).max(axis=1)[:, None, None])
    assert err.max() <= tol, err.max()
    # invalid indices: NaN there, the other entries unchanged
    bad_r, bad_f = rows.copy(), fidx.copy()
    bad_r[-1], bad_f[0] = len(T), len(s)
    b = td.entries(gm, getattr(td, op), f, bad_r, cols, bad_f, prec=getattr(td, prec)).cpu().numpy()
    assert np.isnan(b[:, -1]).all() and np.isnan(b[0]).all()
    assert np.array_equal(b[1:, :-1], g[1:, :-1])
