"""Workloads of the library as a user's program runs them, through its public entry points.

A case is a dict of plain values; prepare() makes what such a program holds
before the call (mesh, frequency set, cluster tree, tensor, right-hand sides),
run() is one call, exact() the same result from a plain FP64 evaluation of the
operators' definition (7-point rule, Sauter-Schwab rule for touching pairs).

Kinds:
  entries     td.entries on rows x cols x frequencies
  compress    td.compress of a prepared mesh and tree, then its first weighted
              apply (how a program gets from a mesh to its first product)
  weighted    Tensor.apply_weighted, sum_l A(s_l) W_l (the history sums of the
              time marching)
  freq        Tensor.apply_freq, one operator A(s_l) x
  solve       Tensor.solve, GMRES on A(s_l) x = b (one time step's system)
  predictor   Model.loss_grad, forward and backward of the rank predictor

Frequency sets: "bdf2" (N points of step dt), "gcq" (contour of 2-stage Radau
IIA over N steps of ratio 1.01 with T = 0.015, as printed), "steps" (the N
pairs (2 -+ i sqrt 2) / dt_n of graded steps, the step operators' points).
"""
import math

import numpy as np
import torch

import paper_2505_00715_gb300 as td
from paper_2505_00715_gb300.inputs import graded_steps, housing, icosphere

OPS = {"slp": td.SLP, "dlp": td.DLP, "adlp": td.ADLP}
SPHERE = dict(mesh="sphere", leaf=32, c=1.0)     # R = 1, triangles 20 * 4^size
HOUSING = dict(mesh="housing", leaf=64, c=343.0)  # machine housing, about `size` triangles


def listed():
    return [
        # a few entries on demand (an error probe, a single coupling): all latency
        dict(HOUSING, name="entries_point", kind="entries", size=2640, op="slp", prec="mixed", freqs="steps", N=4,
             dt=2e-5, nr=5, nc=9, nf=1),
        # the dense reference problem: every entry of the 320-triangle sphere at 16 frequencies, FP64
        dict(SPHERE, name="entries_dense320_fp64", kind="entries", size=2, op="slp", prec="fp64", freqs="bdf2", N=16,
             dt=0.1, nr=320, nc=320, nf=16),
        # a ragged strip of double-layer entries (rows checked against a compressed tensor)
        dict(HOUSING, name="entries_strip_dlp", kind="entries", size=10000, op="dlp", prec="mixed", freqs="steps",
             N=11, dt=2e-5, nr=67, nc=1801, nf=11),
        # mesh to first product in the FP64 form
        dict(SPHERE, name="compress_sphere1280_fp64", kind="compress", size=3, op="slp", prec="fp64", freqs="bdf2",
             N=64, dt=0.05, nrhs=16),
        # the 3D-ACA sphere problem, both layer operators of the direct formulation
        dict(SPHERE, name="compress_sphere5120", kind="compress", size=4, op="slp", prec="mixed", freqs="bdf2", N=64,
             dt=0.05, nrhs=16),
        dict(SPHERE, name="compress_sphere5120_dlp", kind="compress", size=4, op="dlp", prec="mixed", freqs="bdf2",
             N=64, dt=0.05, nrhs=16),
        # the machine housing over the 256-point contour, the benchmark's problem
        dict(HOUSING, name="compress_housing30k", kind="compress", size=30000, op="slp", prec="mixed", freqs="gcq",
             N=256, dt=0.0, nrhs=16),
        # the history sum of one marching step on that tensor, 16 right-hand sides
        dict(HOUSING, name="weighted_housing30k", kind="weighted", size=30000, op="slp", prec="mixed", freqs="gcq",
             N=256, dt=0.0, nrhs=16),
        # the same on a small problem with an odd number of right-hand sides
        dict(SPHERE, name="weighted_sphere1280", kind="weighted", size=3, op="slp", prec="mixed", freqs="bdf2", N=64,
             dt=0.05, nrhs=3),
        # one step operator times one vector (what a Krylov method of the caller runs)
        dict(HOUSING, name="freq_housing30k", kind="freq", size=30000, op="slp", prec="mixed", freqs="steps", N=8,
             dt=2e-5, nrhs=1),
        # one time step's system for four right-hand sides
        dict(SPHERE, name="solve_sphere5120", kind="solve", size=4, op="slp", prec="mixed", freqs="steps", N=4,
             dt=0.1, nrhs=4),
        # one minibatch of the rank predictor's training
        dict(name="predictor_batch4096", kind="predictor", n=4096),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["entries", "entries", "compress", "compress", "weighted", "weighted", "freq", "solve", "predictor"])
    if kind == "predictor":
        return dict(kind=kind, n=_log(rng, 64, 100000))
    op = "slp" if kind == "solve" else rng.choice(["slp", "slp", "dlp", "adlp"])
    prec = "fp64" if rng.random() < 0.25 else "mixed"
    if kind == "entries":
        case = dict(SPHERE, size=rng.choice([2, 3, 4])) if rng.random() < 0.4 else dict(HOUSING, size=_log(rng, 2640, 20000))
        case.update(freqs="steps", N=_log(rng, 1, 24), dt=0.1 if case["mesh"] == "sphere" else 2e-5, nr=_log(rng, 1, 300),
                    nc=_log(rng, 1, 600 if prec == "fp64" else 3000))
        case["nr"], case["nc"] = min(case["nr"], 160), min(case["nc"], 160 if case["size"] == 2 else 3000)
        case["nf"] = rng.randint(1, case["N"])
    else:
        if prec == "fp64":
            case = dict(SPHERE, size=rng.choice([2, 3])) if rng.random() < 0.5 else dict(HOUSING, size=_log(rng, 2640, 3500))
        elif rng.random() < 0.3:
            case = dict(SPHERE, size=rng.choice([3, 4]))
        else:
            case = dict(HOUSING, size=_log(rng, 2640, 20000))
        if kind in ("freq", "solve"):
            case.update(freqs="steps", N=rng.randint(1, 12), dt=(0.1 if case["mesh"] == "sphere" else 2e-5) * rng.uniform(0.5, 2.0))
        elif case["mesh"] == "sphere":
            case.update(freqs="bdf2", N=_log(rng, 7, 64), dt=rng.uniform(0.04, 0.12))
        else:
            case.update(freqs="gcq", N=2 * _log(rng, 8, 32 if prec == "fp64" else 128), dt=0.0)
        case["nrhs"] = _log(rng, 1, 6 if kind == "solve" else 32)
    return dict(case, kind=kind, op=op, prec=prec)


# ---- what a program holds before the call ---------------------------------------
def _mesh(case, seed):
    """Vertices and triangles; the seed moves every vertex by up to 1 % of the mean edge."""
    if case["mesh"] == "housing":
        return housing(case["size"], seed=seed)
    V, T = icosphere(case["size"])
    rng = np.random.default_rng(seed)
    h = np.mean(np.linalg.norm(V[T[:, 0]] - V[T[:, 1]], axis=1))
    d = rng.normal(size=V.shape)
    return V + d * (0.01 * h * rng.random(len(V)) / np.linalg.norm(d, axis=1))[:, None], T


def _points(case):
    """The frequency points (None for the gCQ contour)."""
    if case["freqs"] == "bdf2":
        N = case["N"]
        z = 1e-8 ** (1.0 / (2 * N)) * np.exp(2j * np.pi * np.arange(N) / N)
        return ((1 - z) + (1 - z) ** 2 / 2) / case["dt"]
    if case["freqs"] == "steps":
        dts = case["dt"] * 1.01 ** np.arange(case["N"])
        return np.stack([(2 - 1j * math.sqrt(2)) / dts, (2 + 1j * math.sqrt(2)) / dts], 1).ravel()
    return None


def _freqs(ctx, case):
    if case["freqs"] == "bdf2":
        return td.Freqs.bdf2(ctx, case["N"], case["dt"])
    if case["freqs"] == "steps":
        return td.Freqs.points(ctx, _points(case))
    return td.Freqs.gcq(ctx, graded_steps(case["N"], 1.01, 0.015), td.RADAU2, case["N"], rho=1.0)


def _index(case, seed, ndof, ncol):
    """Rows, columns and frequencies of an entries case: rows near each other and
    columns from all over, as a check of a strip takes them."""
    rng = np.random.default_rng(seed + 1)
    r0 = int(rng.integers(0, ndof - case["nr"] + 1))
    rows = np.arange(r0, r0 + case["nr"], dtype=np.int32)
    cols = rng.permutation(ncol)[:case["nc"]].astype(np.int32)
    return rows, cols, np.arange(case["nf"], dtype=np.int32)


def _gauss(shape, seed, prec, device="cuda"):
    g = torch.Generator(device=device).manual_seed(seed + 2)
    real = torch.randn(shape + (2,), generator=g, device=device, dtype=torch.float64 if prec == "fp64" else torch.float32)
    return torch.view_as_complex(real)


def _samples(case, seed):
    """Features and rank bins of a predictor batch (bins that follow the features)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn(case["n"], 6, generator=g, device="cuda") * torch.tensor([0.8, 0.8, 0.9, 0.3, 1.2, 1.2], device="cuda")
    z = 7.5 + 2.5 * x[:, 0] - 1.5 * x[:, 2] + 2.0 * x[:, 5] + torch.randn(case["n"], generator=g, device="cuda")
    return x, z.round().clamp(0, 15).to(torch.int32)


def prepare(case, seed):
    ctx = td.Context(0)
    if case["kind"] == "predictor":
        x, labels = _samples(case, seed)
        return dict(case=case, model=td.Model(ctx, seed=seed % 1000 + 1), x=x, labels=labels)
    V, T = _mesh(case, seed)
    mesh = td.Mesh(ctx, V, T)
    f = _freqs(ctx, case)
    op, prec = OPS[case["op"]], td.FP64 if case["prec"] == "fp64" else td.MIXED
    colb = td.P1 if case["op"] == "dlp" else td.P0
    s = dict(case=case, ctx=ctx, mesh=mesh, f=f, op=op, prec=prec)
    if case["kind"] == "entries":
        s["rows"], s["cols"], s["fidx"] = _index(case, seed, len(T), mesh.ndof(colb))
        return s
    s["tree"] = td.Tree(mesh, td.P0, colb, case["leaf"], 2.0)
    n = mesh.ndof(colb)
    if case["kind"] in ("compress", "weighted"):
        s["W"] = _gauss((f.NQ, n, case["nrhs"]), seed, case["prec"])
    else:
        s["x"] = _gauss((n, case["nrhs"]), seed, case["prec"])
    if case["kind"] != "compress":
        s["tensor"] = td.compress(mesh, op, f, s["tree"], prec=prec, c=case["c"])
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "entries":
        return td.entries(s["mesh"], s["op"], s["f"], s["rows"], s["cols"], s["fidx"], prec=s["prec"], c=case["c"])
    if kind == "compress":
        return td.compress(s["mesh"], s["op"], s["f"], s["tree"], prec=s["prec"], c=case["c"]).apply_weighted(s["W"])
    if kind == "weighted":
        return s["tensor"].apply_weighted(s["W"])
    if kind == "freq":
        return s["tensor"].apply_freq(_fidx(case), s["x"])
    if kind == "solve":
        return s["tensor"].solve(_fidx(case), s["x"], tol=1e-10 if case["prec"] == "fp64" else 1e-6, maxit=400, check=False)[0]
    loss, grad = s["model"].loss_grad(s["x"], s["labels"])
    return {"loss": loss, "grad": grad}


def _fidx(case):
    return 2 * (case["N"] // 2)


# ---- work ------------------------------------------------------------------------
def _counts(case):
    """Rows, columns, frequency points and unique ones."""
    nt = 20 * 4 ** case["size"] if case["mesh"] == "sphere" else case["size"]
    NQ = 2 * case["N"] if case["freqs"] == "steps" else case["N"]
    Nu = NQ // 2 + 1 if case["freqs"] == "bdf2" else NQ // 2
    return nt, nt // 2 if case["op"] == "dlp" else nt, NQ, Nu


def work(case):
    """Bytes and operations of one pass, as estimates from the sizes alone: a point
    pair costs 25 operations per frequency, an entry 49 point pairs (a P1 column 6
    times as many); a compressed tensor keeps 14 leaves' columns per row near and
    140 face values per row and level and 8 terms far."""
    if case["kind"] == "predictor":
        return {"bytes": 28.0 * case["n"] + 8 * 5648, "flops": 6.0 * 5504 * case["n"]}
    es = 16 if case["prec"] == "fp64" else 8
    nt, ncol, NQ, Nu = _counts(case)
    per = 25.0 * 49 * (6 if case["op"] == "dlp" else 1)
    if case["kind"] == "entries":
        n = float(case["nr"]) * case["nc"] * case["nf"]
        return {"bytes": es * n, "flops": per * n}
    near = nt * min(ncol, 14 * case["leaf"])
    faces = 8.0 * near + 8.0 * 140 * nt * math.log2(max(2.0, nt / case["leaf"]))
    q = case.get("nrhs", 1)
    vec = es * q * (NQ * ncol + nt)
    one = es * q * (ncol + nt)
    if case["kind"] == "compress":
        return {"bytes": es * faces + vec, "flops": per * (near * Nu + 2 * faces) + 16.0 * q * faces}
    if case["kind"] == "weighted":
        return {"bytes": es * faces + vec, "flops": 16.0 * q * faces}
    if case["kind"] == "freq":
        return {"bytes": es * faces + one, "flops": 8.0 * q * faces}
    return {"bytes": 15 * (es * faces + one), "flops": 15 * 8.0 * q * faces}


# ---- FP64 evaluation of the definition -----------------------------------------------
# barycentric points and weights of the 7-point degree-5 rule
def _rule7():
    q = math.sqrt(15.0)
    pts, wts = [(1 / 3, 1 / 3, 1 / 3)], [9 / 40]
    for a, w in (((6 - q) / 21, (155 - q) / 1200), ((6 + q) / 21, (155 + q) / 1200)):
        pts += [(a, a, 1 - 2 * a), (a, 1 - 2 * a, a), (1 - 2 * a, a, a)]
        wts += [w] * 3
    return np.array(pts), np.array(wts)


class _Exact:
    """Operator values on the mesh V, T for sigma = s / c, in float64."""

    def __init__(self, V, T, op, device):
        self.op, self.dev, self.T = op, device, T
        t = lambda a: torch.as_tensor(a, dtype=torch.float64, device=device)  # noqa: E731
        self.bary, w = _rule7()
        P = V[T]
        n = np.cross(P[:, 1] - P[:, 0], P[:, 2] - P[:, 0])
        dbl = np.linalg.norm(n, axis=1)
        self.P, self.N, self.dbl = P, n / dbl[:, None], dbl
        self.x = t(np.einsum("qk,tkc->tqc", self.bary, P))
        self.w = t(0.5 * dbl[:, None] * w)
        self.n, self.hat = t(self.N), t(self.bary)

    def kernel(self, r, dn, sigma):
        """e^{-sigma r} / r, or (1 + sigma r) e^{-sigma r} dn / r^3, real and imaginary part."""
        e = torch.exp(-sigma.real * r)
        f = e / r if self.op == "slp" else e * dn / (r * r * r)
        c, s = torch.cos(sigma.imag * r), torch.sin(sigma.imag * r)
        if self.op == "slp":
            return f * c, -f * s
        p, q = 1 + sigma.real * r, sigma.imag * r
        return f * (p * c + q * s), f * (q * c - p * s)

    def regular(self, rows, tris, sigmas):
        """[nf][rows][tris][1 or 3] by the 7-point rule (touching pairs hold nothing)."""
        d = self.x[tris][None, :, None] - self.x[rows][:, None, :, None]  # y - x: row, tri, qx, qy
        r = d.square().sum(-1).sqrt()
        dn = None
        if self.op == "dlp":
            dn = -torch.einsum("rtabc,tc->rtab", d, self.n[tris])
        elif self.op == "adlp":
            dn = torch.einsum("rtabc,rc->rtab", d, self.n[rows])
        wx, wy = self.w[rows], self.w[tris]
        touch = torch.as_tensor(self.touching(rows, tris), device=self.dev)
        r = torch.where(touch[:, :, None, None], torch.ones_like(r), r)
        out = []
        for sg in sigmas:
            v = [torch.einsum("rtab,ra,tb->rtb", k, wx, wy) for k in self.kernel(r, dn, sg)]
            v = [torch.where(touch[:, :, None], torch.zeros_like(k), k) for k in v]
            v = [k @ self.hat if self.op == "dlp" else k.sum(-1, keepdim=True) for k in v]
            out.append(torch.complex(v[0], v[1]) / (4 * math.pi))
        return torch.stack(out)

    def touching(self, rows, tris):
        a, b = self.T[rows.cpu().numpy()], self.T[tris.cpu().numpy()]
        hit = np.zeros((len(a), len(b)), dtype=bool)
        for i in range(3):
            for j in range(3):
                hit |= a[:, i][:, None] == b[None, :, j]
        return hit

    def singular(self, ti, tj, sigmas, ng=5):
        """[nf][pairs][1 or 3] of touching pairs (ti[k], tj[k]) by the Sauter-Schwab rule."""
        if self.op == "slp":
            ti, tj = np.minimum(ti, tj), np.maximum(ti, tj)
        same = self.T[ti][:, :, None] == self.T[tj][:, None, :]
        shared = same.sum((1, 2))
        out = torch.zeros(len(sigmas), len(ti), 3 if self.op == "dlp" else 1, dtype=torch.complex128, device=self.dev)
        x, w = np.polynomial.legendre.leggauss(ng)
        x, w = 0.5 * (x + 1), 0.5 * w
        for cls in (1, 2, 3):
            at = np.nonzero(shared == cls)[0]
            if not len(at) or (cls == 3 and self.op != "slp"):
                continue  # a flat panel's double layer on itself is zero
            la, lb = self.order(cls, same[at])
            P = np.take_along_axis(self.P[ti[at]], la[:, :, None], 1)
            Q = np.take_along_axis(self.P[tj[at]], lb[:, :, None], 1)
            coef, wt, lam = getattr(self, "rule%d" % cls)(x, w)
            # y - x = coef . (P1 - P0, P2 - P1, Q1 - Q0, Q2 - Q1)
            E = np.stack([P[:, 1] - P[:, 0], P[:, 2] - P[:, 1], Q[:, 1] - Q[:, 0], Q[:, 2] - Q[:, 1]], 1)
            for c0 in range(0, len(at), 2048):
                sl = slice(c0, c0 + 2048)
                d = np.einsum("qe,pec->pqc", coef, E[sl])
                dn = None
                if self.op == "dlp":
                    dn = -np.einsum("pqc,pc->pq", d, self.N[tj[at[sl]]])
                elif self.op == "adlp":
                    dn = np.einsum("pqc,pc->pq", d, self.N[ti[at[sl]]])
                g = self.dbl[ti[at[sl]]] * self.dbl[tj[at[sl]]]
                to = lambda a: None if a is None else torch.as_tensor(a, device=self.dev)  # noqa: E731
                r, dn, wq = to(np.linalg.norm(d, axis=2)), to(dn), to(wt[None] * g[:, None])
                idx = torch.as_tensor(at[sl], device=self.dev)
                for k, sg in enumerate(sigmas):
                    re, im = self.kernel(r, dn, sg)
                    v = torch.complex(re * wq, im * wq) / (4 * math.pi)
                    if self.op == "dlp":
                        v = v @ to(lam).to(v.dtype)  # in the order of the parametrisation
                        out[k, idx[:, None], to(lb[sl])] = v
                    else:
                        out[k, idx, 0] = v.sum(1)
        return out

    @staticmethod
    def order(cls, same):
        """Local vertex order of both triangles: shared vertices first (a common edge
        in the order of the first triangle's vertices), or cyclic from the shared one."""
        n = len(same)
        if cls == 3:
            return np.tile(np.arange(3), (n, 1)), np.tile(np.arange(3), (n, 1))
        a, b = same.any(2), same.argmax(2)
        if cls == 1:
            i = a.argmax(1)
            return (i[:, None] + np.arange(3)) % 3, (b[np.arange(n), i][:, None] + np.arange(3)) % 3
        off = (~a).argmax(1)
        i0, i1 = np.where(off == 0, 1, 0), np.where(off == 2, 1, 2)
        j0, j1 = b[np.arange(n), i0], b[np.arange(n), i1]
        return np.stack([i0, i1, 3 - i0 - i1], 1), np.stack([j0, j1, 3 - j0 - j1], 1)

    # Points of the transformed integrals: difference coefficients, weights
    # (Jacobian (2|ti|)(2|tj|) left out) and the trial point's barycentrics.
    @staticmethod
    def rule3(x, w):
        rays = np.array([[1, 0], [1, 1], [0, 1], [-1, 0], [-1, -1], [0, -1]], dtype=np.float64)
        coef, wt = [], []
        for k in range(6):
            for a, wa in zip(x, w):
                for b, wb in zip(x, w):
                    z = a * (rays[k] + b * (rays[(k + 1) % 6] - rays[k]))
                    coef.append([z[0], z[1], 0, 0])  # both triangles are one: z in its own edges
                    wt.append(wa * wb * a * (1 - a) ** 2 / 2)
        return np.array(coef), np.array(wt), None

    @staticmethod
    def rule2(x, w):
        cones = np.array([[[0, 1, 0], [1, 0, 0], [1, 0, 1]], [[0, 1, 0], [1, 0, 1], [0, 1, 1]],
                          [[0, 0, 1], [1, 0, 1], [0, 1, 1]], [[0, 1, 0], [0, 1, 1], [-1, 1, 0]],
                          [[-1, 0, 0], [0, 0, 1], [0, 1, 1]], [[-1, 0, 0], [0, 1, 1], [-1, 1, 0]]], dtype=np.float64)
        coef, wt, lam = [], [], []
        for A, B, C in cones:
            for a, wa in zip(x, w):
                for b, wb in zip(x, w):
                    for c, wc in zip(x, w):
                        u, p, q = a * (A + b * (B - A) + b * c * (C - B))
                        coef.append([u, -p, 0, q])  # the common edge is P1 - P0
                        wt.append(wa * wb * wc * a * a * b * (1 - a))
                        mid = 0.5 * (max(p, q - u) + (1 - u if u > 0 else 1.0))
                        lam.append([1 - mid - u, mid + u - q, q])
        return np.array(coef), np.array(wt), np.array(lam)

    @staticmethod
    def rule1(x, w):
        coef, wt, lam = [], [], []
        for swap in (False, True):
            for a, wa in zip(x, w):
                for b, wb in zip(x, w):
                    for c, wc in zip(x, w):
                        for e, we in zip(x, w):
                            big, small = (a, a * b), (a * c, a * c * e)
                            X, Y = (small, big) if swap else (big, small)
                            coef.append([-X[0], -X[1], Y[0], Y[1]])
                            wt.append(wa * wb * wc * we * a ** 3 * c)
                            lam.append([1 - Y[0], Y[0] - Y[1], Y[1]])
        return np.array(coef), np.array(wt), np.array(lam)

    def touching_pairs(self, rows):
        """All touching (row position, triangle) pairs of the rows."""
        nv = int(self.T.max()) + 1
        around = [[] for _ in range(nv)]
        for t, tri in enumerate(self.T):
            for v in tri:
                around[v].append(t)
        got = [(i, t) for i, r in enumerate(rows) for t in sorted({t for v in self.T[r] for t in around[v]})]
        return np.array(got, dtype=np.int64).reshape(-1, 2)

    def blocks(self, rows, sigmas):
        """(row positions, [nf][rows][all triangles][1 or 3]) in runs of rows."""
        nt = len(self.T)
        step = max(1, (1 << 24) // (49 * nt))
        tp = self.touching_pairs(rows)
        for r0 in range(0, len(rows), step):
            rr = torch.as_tensor(rows[r0:r0 + step], dtype=torch.int64, device=self.dev)
            A = self.regular(rr, torch.arange(nt, device=self.dev), sigmas)
            mine = tp[(tp[:, 0] >= r0) & (tp[:, 0] < r0 + step)]
            v = self.singular(rows[mine[:, 0]], mine[:, 1], sigmas)
            A[:, torch.as_tensor(mine[:, 0] - r0, device=self.dev), torch.as_tensor(mine[:, 1], device=self.dev)] = v
            yield slice(r0, r0 + len(rr)), A

    def dofs(self, A):
        """Triangle values [.., tris, 1 or 3] to columns (P1: summed around every vertex)."""
        if self.op != "dlp":
            return A[..., 0]
        nv = int(self.T.max()) + 1
        out = torch.zeros(A.shape[:-2] + (nv,), dtype=A.dtype, device=self.dev)
        for k in range(3):
            out.index_add_(-1, torch.as_tensor(self.T[:, k].astype(np.int64), device=self.dev), A[..., k].contiguous())
        return out


def _exact_cost(case, rows, nu):
    return 49.0 * rows * _counts(case)[0] * nu


def exact(case, seed):
    if case["kind"] == "predictor":
        return _exact_predictor(case, seed)
    if case["freqs"] == "gcq":
        return None  # the contour's points come from elliptic functions
    s = _points(case) / case["c"]
    V, T = _mesh(case, seed)
    E = _Exact(V, np.asarray(T, dtype=np.int64), case["op"], "cuda" if torch.cuda.is_available() else "cpu")
    nt = len(T)
    if case["kind"] == "entries":
        rows, cols, fidx = _index(case, seed, nt, len(V) if case["op"] == "dlp" else nt)
        if _exact_cost(case, len(rows), len(fidx)) > 5e10:
            return None
        out = [E.dofs(A)[:, :, torch.as_tensor(cols.astype(np.int64), device=E.dev)] for _, A in E.blocks(rows.astype(np.int64), s[fidx])]
        return torch.cat(out, 1)
    every = np.arange(nt)
    if case["kind"] in ("freq", "solve"):
        if _exact_cost(case, nt, 1) > 6e10:
            return None
        x = _gauss((len(V) if case["op"] == "dlp" else nt, case["nrhs"]), seed, case["prec"]).to(torch.complex128)
        s1 = s[[_fidx(case)]]
        if case["kind"] == "freq":
            return torch.cat([E.dofs(A)[0] @ x for _, A in E.blocks(every, s1)])
        if nt > 6000:
            return None
        return torch.linalg.solve(torch.cat([E.dofs(A)[0] for _, A in E.blocks(every, s1)]), x)
    keep = np.nonzero(s.imag >= -1e-9 * np.abs(s))[0]  # one of each conjugate pair
    if _exact_cost(case, nt, len(keep)) > 6e10:
        return None
    NQ = len(s)
    W = _gauss((NQ, len(V) if case["op"] == "dlp" else nt, case["nrhs"]), seed, case["prec"]).to(torch.complex128)
    y = torch.zeros(nt, case["nrhs"], dtype=torch.complex128, device=E.dev)
    for at, A in E.blocks(every, s[keep]):
        A = E.dofs(A)
        for k, q in enumerate(keep):
            y[at] += A[k] @ W[q]
            if (NQ - q) % NQ != q:
                y[at] += A[k].conj() @ W[(NQ - q) % NQ]
    return y


def _exact_predictor(case, seed):
    x, labels = _samples(case, seed)
    p = torch.as_tensor(td.Model(td.Context(0), seed=seed % 1000 + 1).params(), dtype=torch.float64, device="cuda").requires_grad_()
    W1, b1, W2, b2, W3, b3 = torch.split(p, [384, 64, 4096, 64, 1024, 16])
    g = torch.nn.functional.gelu
    h = g(x.double() @ W1.view(64, 6).T + b1)
    h = g(h @ W2.view(64, 64).T + b2)
    loss = torch.nn.functional.cross_entropy(h @ W3.view(16, 64).T + b3, labels.long())
    loss.backward()
    return {"loss": loss.detach().view(1), "grad": p.grad}
