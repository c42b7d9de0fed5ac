"""FP64 entries at the edges of the table-driven exponential (run with -m gpu):
tiny and large |s| r, the library branch beyond Re s r = 704 and |Im s| r = 65536,
and points around both limits, for the kernels that evaluate single exponentials
(near table, generic entries, and far fibres at pairs that do not touch, the only
ones they are meant for), against the FP64 oracle.

Tolerance, of an entry's sum of moduli: 1e-12 (as the entry paths are held to) and
4e-15 |s|: coordinates and r <= 2 are good to a few 2^-53 on either side, which the
phase s r multiplies by |s|.
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


@pytest.mark.parametrize("op", ["SLP", "DLP", "ADLP"])
@pytest.mark.parametrize("path", ["PATH_GENERIC", "PATH_NEAR", "PATH_FIBRE"])
@pytest.mark.parametrize("s", [1e-9, 0.02 + 0.01j, 3 - 40j, 300 + 900j, 360 + 2j, 0.5 + 33000j, 0.1 - 60000j, 2000 + 3e5j])
def test_exponential_ranges(td, ctx, orc, op, path, s):
    V, T = icosphere(1)
    gm, om = td.Mesh(ctx, V, T), orc.Mesh(V, T)
    f = td.Freqs.points(ctx, np.array([s], dtype=np.complex128))
    rows = np.arange(0, len(T), 3, dtype=np.int32)
    cols = np.arange(len(V) if op == "DLP" else len(T), dtype=np.int32)
    g = td.entries(gm, getattr(td, op), f, rows, cols, [0], prec=td.FP64, path=getattr(td, path)).cpu().numpy()
    ng = 5
    o = om.entries(getattr(orc, op), rows, cols, [s], ng=ng)
    mag = om.entries_mag(getattr(orc, op), rows, cols, [s], ng=ng)
    err = np.abs(g - o) / np.maximum(mag, 1e-6 * mag.max())
    if path == "PATH_FIBRE":
        vert = np.zeros((len(T), len(V)), dtype=bool)
        vert[np.arange(len(T))[:, None], T] = True
        touch = vert.astype(int) @ vert.T.astype(int) > 0  # triangle pairs
        if op == "DLP":
            touch = touch.astype(int) @ vert.astype(int) > 0  # with any triangle of the column's support
        err = err[:, ~touch[np.ix_(rows, cols)]]
    assert err.max() <= 1e-12 + 4e-15 * abs(s), err.max()
