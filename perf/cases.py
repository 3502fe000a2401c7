"""The work that the library is timed on: whole runs of implicit steps, single linear solves,
condensations and post-processings, each through the public entry points of `hdg.Solver`.

`listed()` names the cases, `draw()` gives more of the same ranges, `prepare()` builds what a
program holds before the call (mesh, material, solver, condensed operators, initial state),
`run()` is one pass, `work()` its unavoidable bytes and operations, and `exact()` the same
outputs from a plain 64-bit formulation below that shares no code with the library: dense
element blocks by quadrature, pivoted LU, and a trace solve to the last digits.

A pass of the marching cases sets the initial state and advances `steps` implicit steps, so
every pass does the same work; materials, sources and initial fields come from the seed.
"""
import itertools
import math

import numpy as np
import torch

from paper_1807_00086_gb300 import hdg, inputs

T_START = 0.1            # the sources (peak at 0.12) are rising when a marching case begins
F0, T0 = 10.0, 0.12      # Ricker wavelet of every source


def listed():
    return [
        # the 2D first example of a user: 512 triangles, every kernel far smaller than the GPU
        {"name": "square_be_k2", "kind": "march", "dim": 2, "N": 16, "k": 2, "prec": "fp64", "scheme": "be",
         "R": 1, "dt": 0.01, "steps": 50},
        # the headline workload: 196,608 tetrahedra, FP16 operator, BDF2
        {"name": "cube_bdf2_k3", "kind": "march", "dim": 3, "N": 32, "k": 3, "prec": "mixed16", "scheme": "bdf2",
         "R": 1, "dt": 2e-3, "steps": 12},
        # the default precision of the solver on a mid-sized mesh of odd side
        {"name": "cube_bdf2_k2_fp64", "kind": "march", "dim": 3, "N": 19, "k": 2, "prec": "fp64", "scheme": "bdf2",
         "R": 1, "dt": 2e-3, "steps": 10},
        # two shapes of the serving ladder with the serving width of four columns
        {"name": "serve_square_k2", "kind": "march", "dim": 2, "N": 45, "k": 2, "prec": "mixed", "scheme": "bdf2",
         "R": 4, "dt": 2e-3, "steps": 16},
        {"name": "serve_cube_k3", "kind": "march", "dim": 3, "N": 14, "k": 3, "prec": "mixed", "scheme": "bdf2",
         "R": 4, "dt": 2e-3, "steps": 10},
        # many sources in one medium: 64 columns on one operator
        {"name": "sources64_k3", "kind": "march", "dim": 3, "N": 16, "k": 3, "prec": "mixed", "scheme": "bdf2",
         "R": 64, "dt": 2e-3, "steps": 8},
        # elastic waves, a degree per element, DIRK(3,3)
        {"name": "elastic_mixed_degree", "kind": "elastic", "N": 16, "k": 0, "prec": "mixed16", "dt": 1e-3, "steps": 4},
        # elastic waves, one degree, odd mesh side
        {"name": "elastic_k2", "kind": "elastic", "N": 11, "k": 2, "prec": "mixed", "dt": 1e-3, "steps": 4},
        # a change of the time step: all element blocks condensed again, and the Schur blocks read back
        {"name": "condense_k3", "kind": "condense", "dim": 3, "N": 24, "k": 3, "prec": "mixed16"},
        # one linear system given by the caller: condensed right-hand side, trace solve, recovery
        {"name": "linear_solve_k3", "kind": "solve", "dim": 2, "N": 91, "k": 3, "prec": "mixed"},
        # nonlinear plate: a Newton condensation per iteration
        {"name": "svk_plate_k2", "kind": "svk", "N": 16, "k": 2, "prec": "mixed", "dt": 2e-3, "steps": 1},
        # an output time: the superconvergent pressure of every element
        {"name": "postprocess_k3", "kind": "post", "dim": 3, "N": 27, "k": 3},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _simplices(dim, N):
    return 2 * N * N if dim == 2 else 6 * N ** 3


def _cap(dim, entries, per_elem):
    """largest N whose elements x per_elem stays within `entries` (2D: up to 131,072 triangles)"""
    ne = entries / per_elem
    return max(1, min(256, int(math.sqrt(ne / 2)))) if dim == 2 else max(1, int((ne / 6) ** (1.0 / 3.0)))


def draw(rng):
    kind = rng.choice(["march", "march", "columns", "columns", "sources", "elastic", "elastic", "condense", "solve",
                       "svk", "post"])
    dim = rng.choice([2, 3])
    k = rng.randint(1, 4)
    if kind in ("march", "columns", "condense", "solve", "post"):
        n, m = _n_m(dim, k)
    lo = 8 if dim == 2 else 3
    if kind == "march":
        prec = rng.choice(["fp64", "mixed", "mixed16", "mixed16"])
        hi = _cap(dim, 2.0e6 if prec == "fp64" else 1.2e7, n)
        return {"kind": "march", "dim": dim, "N": _log_int(rng, lo, hi), "k": k, "prec": prec,
                "scheme": rng.choice(["be", "bdf2", "bdf2"]), "R": 1, "dt": rng.choice([2e-3, 5e-3]),
                "steps": rng.randint(6, 12)}
    if kind == "columns":
        R = rng.choice([2, 4, 4, 8])
        hi = _cap(dim, 8.0e6 / R, n)
        return {"kind": "march", "dim": dim, "N": _log_int(rng, lo, hi), "k": k, "prec": "mixed", "scheme": "bdf2",
                "R": R, "dt": 2e-3, "steps": rng.randint(6, 12)}
    if kind == "sources":
        k, R = rng.choice([2, 3]), rng.choice([32, 64])
        hi = _cap(3, 1.0e8 / R, _n_m(3, k)[0])
        return {"kind": "march", "dim": 3, "N": _log_int(rng, 3, hi), "k": k, "prec": "mixed", "scheme": "bdf2",
                "R": R, "dt": 2e-3, "steps": rng.randint(4, 8)}
    if kind == "elastic":
        k = rng.choice([0, 0, 1, 2, 3])
        hi = {0: 16, 1: 20, 2: 15, 3: 12}[k]
        return {"kind": "elastic", "N": _log_int(rng, 3, hi), "k": k,
                "prec": rng.choice(["mixed", "mixed16"]) if k == 0 else "mixed", "dt": 1e-3, "steps": rng.randint(2, 4)}
    if kind == "condense":
        hi = _cap(dim, 1.3e8, m * m)
        return {"kind": "condense", "dim": dim, "N": _log_int(rng, lo, hi), "k": k,
                "prec": rng.choice(["fp64", "mixed", "mixed16"])}
    if kind == "solve":
        prec = rng.choice(["fp64", "mixed", "mixed16"])
        hi = _cap(dim, 2.0e6, n)
        return {"kind": "solve", "dim": dim, "N": _log_int(rng, lo, hi), "k": k, "prec": prec}
    if kind == "svk":
        k = rng.choice([1, 2, 2])
        return {"kind": "svk", "N": _log_int(rng, 4, 16), "k": k, "prec": "mixed", "dt": 2e-3, "steps": 1}
    hi = _cap(dim, 8.0e6, n)
    return {"kind": "post", "dim": dim, "N": _log_int(rng, lo, hi), "k": k}


def _n_m(dim, k):
    """field and trace entries of an acoustic element"""
    return (dim + 1) * math.comb(k + dim, dim), (dim + 1) * math.comb(k + dim - 1, dim - 1)


def work(case):
    """Bytes: fields and traces in and out, and each stored operator once per implicit stage.
    Operations: one S_K product, one condensed right-hand side and one recovery per stage (the
    condensation and the post-processing: their dense element algebra)."""
    kind, k = case["kind"], case["k"]
    if kind == "svk":
        ne, Np, nf = 6 * case["N"] ** 2, math.comb(k + 3, 3), 12 * math.comb(k + 2, 2)
        nv = 3 * Np
        stages = 3 * case["steps"]
        flops = stages * 2.0 * ne * (nv ** 3 / 3 + nv * nv * nf + nv * nf * nf)
        return {"bytes": ne * 21 * Np * 16.0 * stages, "flops": flops}
    if kind == "elastic":
        ne = 6 * case["N"] ** 3
        ks = [k] if k else [1, 2, 3, 4]
        word = 2 if case["prec"] == "mixed16" else 4
        b = f = 0.0
        for kk in ks:
            Np, m = math.comb(kk + 3, 3), 12 * math.comb(kk + 2, 2)
            b += ne / len(ks) * (9 * Np * 16 + m * 16 + m * m * word + 9 * Np * Np * 8)
            f += ne / len(ks) * (2 * m * m + 4 * 9 * Np * Np + 8 * 9 * Np * m)
        return {"bytes": 3 * case["steps"] * b, "flops": 3 * case["steps"] * f}
    dim = case["dim"]
    ne = _simplices(dim, case["N"])
    n, m = _n_m(dim, k)
    Np = n // (dim + 1)
    if kind == "condense":
        word = {"fp64": 8, "mixed": 12, "mixed16": 14}[case["prec"]]
        return {"bytes": ne * (m * m * (8 + word) + Np * Np * 8.0),
                "flops": 2.0 * ne * (Np ** 3 / 3 + Np * Np * m / 2 + Np * m * m / 2)}
    if kind == "post":
        n1 = math.comb(k + 1 + dim, dim)
        return {"bytes": ne * 8.0 * (Np + m / 2 + n1), "flops": 2.0 * ne * (n1 ** 3 / 6 + n1 * n1 + dim * Np * (Np + m + n1))}
    R = case.get("R", 1)
    stages = case.get("steps", 1)
    word = {"fp64": 8, "mixed": 4, "mixed16": 2}[case["prec"]]
    bytes_ = ne * (R * (n * 24 + m * 8) + m * (m + 1) / 2 * word + Np * Np * 8)
    return {"bytes": float(stages * bytes_), "flops": float(stages * ne * R * (2 * m * m + 4 * Np * Np + 4 * dim * Np * (Np + m)))}


# ----------------------------------------------------------------------------- inputs

def _mesh(case):
    if case["kind"] == "svk":
        return inputs.plate_tet(case["N"])
    return inputs.unit_cube_tet(case["N"]) if case.get("dim", 3) == 3 else inputs.unit_square_tri(case["N"])


def _alpha(case):
    if case["kind"] == "elastic":
        return 1.0 / (_dirk3()[0][0, 0] * case["dt"])
    return {"be": 1.0, "bdf2": 1.5}[case.get("scheme", "bdf2")] / case.get("dt", 2e-3)


def _data(case, seed):
    """everything of a case that its seed decides (the degrees of a mixed-degree mesh are part of the
    workload, like the mesh: the layouts follow them)"""
    vert, elem = _mesh(case)
    ne = elem.shape[0]
    d = {"vert": vert, "elem": elem, "rho": np.ones(ne)}
    kind = case["kind"]
    if kind == "elastic":
        d["lam"], d["mu"] = inputs.lognormal(ne, 1.5, 0.5, seed), inputs.lognormal(ne, 1.0, 0.5, seed + 1)
        d["elem_k"] = inputs.element_degrees(ne, 1, 4, inputs.DEFAULT_SEED + 7) if case["k"] == 0 else None
        d["center"] = inputs.uniform_points(1, 3, 0.4, 0.6, seed + 3)[0]
        return d
    if kind == "svk":
        d["amp"] = float(np.random.default_rng(seed).uniform(0.3, 0.4))
        return d
    d["c"] = inputs.loguniform(ne, 1.0, 3.0, seed)
    n, m = _n_m(case["dim"], case["k"])
    if kind == "march":
        R = case["R"]
        d["src"] = inputs.uniform_points(R, case["dim"], 0.1, 0.9, seed + 64)
        d["delay"] = np.random.default_rng(seed + 65).uniform(0.0, 0.01, R)
    elif kind == "condense":
        d["x"] = inputs.random_traces(_n_faces(case), m // (case["dim"] + 1), seed + 2)
    elif kind == "solve":
        d["F"] = inputs.random_state(ne, n, seed + 2)
    else:
        d["u"] = inputs.random_state(ne, n, seed + 2)
        d["lam"] = inputs.random_traces(_n_faces(case), m // (case["dim"] + 1), seed + 3)
    return d


def _n_faces(case):
    N = case["N"]
    return 3 * N * N + 2 * N if case["dim"] == 2 else 12 * N ** 3 + 6 * N * N


def _bump(xq, center, comps):
    return inputs.gaussian_velocity_values(xq, center, 0.05, comps)


def prepare(case, seed):
    d = _data(case, seed)
    st = {"case": case}
    dev = lambda a: torch.tensor(a, device="cuda")
    kind = case["kind"]
    if kind == "svk":
        ne = d["elem"].shape[0]
        s = hdg.Solver(d["vert"], d["elem"], case["k"], 1.0, 1.0, lam=np.full(ne, 1.5), mu=np.ones(ne), svk=True,
                       rtol=1e-10, prec=case["prec"])
        zb = s.hdg_quadrature_points(1)[:, :, 2]
        s.hdg_svk_set_traction_faces(np.all(np.abs(zb - 0.01) < 1e-13, axis=1) | np.all(np.abs(zb) < 1e-13, axis=1))
        xv = s.hdg_quadrature_points(0)
        vals = np.zeros(xv.shape[:2] + (21,))
        vals[:, :, 2] = d["amp"] * np.pi * np.sin(np.pi * xv[:, :, 0]) * np.sin(np.pi * xv[:, :, 1])
        st["u0"] = s.hdg_project_volume(vals)
    elif kind == "elastic":
        s = hdg.Solver(d["vert"], d["elem"], case["k"] or 4, 1.0, d["rho"], lam=d["lam"], mu=d["mu"],
                       prec=case["prec"], rtol=1e-12, inner_rtol=1e-3 if case["prec"] == "mixed16" else 3e-6,
                       elem_k=d["elem_k"])
        st["u0"] = s.hdg_project_volume(_bump(s.hdg_quadrature_points(0), d["center"], 9))
        s.hdg_condense(_alpha(case))
    else:
        R, prec = case.get("R", 1), case.get("prec", "fp64")
        inner = {"fp64": None, "mixed": 1e-4 if R > 1 else 3e-6, "mixed16": 1e-3}[prec]
        s = hdg.Solver(d["vert"], d["elem"], case["k"], 1.0, d["rho"], d["c"], prec=prec,
                       rtol=1e-13 if prec == "fp64" else 1e-12, inner_rtol=inner, nrhs=R, use_graphs=R > 1)
        if kind == "march":
            s.hdg_set_sources(d["src"], np.ones(R), F0, T0, col=np.arange(R, dtype=np.int32), delay=d["delay"])
            s.hdg_set_dirichlet(None)
            st["u0"] = s.empty_fields()
            s.hdg_condense(_alpha(case))
        elif kind == "condense":
            st["x"], st["y"] = dev(d["x"]), s.empty_traces()
        elif kind == "solve":
            st["F"], st["r"], st["lam"], st["u"] = dev(d["F"]), s.empty_traces(), s.empty_traces(), s.empty_fields()
            s.hdg_condense(_alpha(case))
        else:
            st["u"], st["lam"] = dev(d["u"]), dev(d["lam"])
            st["p"] = torch.zeros((s.n_elem, math.comb(case["k"] + 1 + s.dim, s.dim)), dtype=torch.float64, device="cuda")
    if kind in ("march", "elastic", "svk"):
        st["u"], st["lam"] = s.empty_fields(), s.empty_traces()
    st["s"] = s
    return st


def run(st):
    case, s = st["case"], st["s"]
    kind = case["kind"]
    if kind in ("march", "elastic", "svk"):
        s.hdg_set_state(st["u0"], T_START)
        s.hdg_step(case["dt"], case.get("scheme", "dirk3"), case["steps"])
        u, lam, _ = s.hdg_get_state(u=st["u"], lam=st["lam"])
        return {"u": u, "lam": lam}
    if kind == "condense":
        s.hdg_condense(_alpha(case))
        return {"S": s.hdg_get_schur(), "y": s.hdg_trace_apply(st["x"], st["y"])}
    if kind == "solve":
        r = s.hdg_condensed_rhs(st["F"], None, st["r"])
        st["lam"].zero_()
        s.hdg_trace_solve(r, st["lam"])
        return {"r": r, "lam": st["lam"], "u": s.hdg_recover(st["F"], st["lam"], st["u"])}
    return {"p": s.hdg_postprocess(st["u"], st["lam"], st["p"])}


# ----------------------------------------------------------------------------- the same in plain 64-bit arithmetic

def exact(case, seed):
    """The outputs of run() from dense element blocks. The nonlinear plate has none: a plain
    Newton solution of it takes minutes."""
    if case["kind"] == "svk":
        return None
    with torch.no_grad():
        return _Plain(case, _data(case, seed)).answer()


def _dirk3():
    """Alexander's SDIRK: (a, b, c)"""
    g = [r.real for r in np.roots([1.0, -3.0, 1.5, -1.0 / 6.0]) if abs(r.imag) < 1e-12 and 1 / 3 < r.real < 0.5][0]
    b1, b2 = -(6 * g * g - 16 * g + 1) / 4, (6 * g * g - 20 * g + 5) / 4
    return np.array([[g, 0, 0], [(1 - g) / 2, g, 0], [b1, b2, g]]), np.array([b1, b2, g]), np.array([g, (1 + g) / 2, 1.0])


def _jacobi(n, a, x):
    """P_n^(a, 0) by its three-term recurrence"""
    p0, p1 = np.ones_like(x), (a + (a + 2) * x) / 2
    if n == 0:
        return p0
    for j in range(1, n):
        c = 2 * j + a
        p0, p1 = p1, ((c + 1) * (c * (c + 2) * x + a * a) * p1 - 2 * (j + a) * j * (c + 2) * p0) / (2 * (j + 1) * (j + a + 1) * c)
    return p1


def _modes(dim, k):
    return [i for i in itertools.product(range(k + 1), repeat=dim) if sum(i) <= k]


def _phi(dim, k, pts):
    """orthonormal Dubiner modes at points of the unit simplex (any analytic argument)"""
    if dim == 1:
        return np.stack([math.sqrt(2 * i + 1) * _jacobi(i, 0, 2 * pts[:, 0] - 1) for (i,) in _modes(1, k)], axis=1)
    if dim == 2:
        x, y = pts.T
        w = 1 - y
        return np.stack([math.sqrt(2.0 * (2 * i + 1) * (i + j + 1)) * _jacobi(i, 0, 2 * x / w - 1) * w ** i
                         * _jacobi(j, 2 * i + 1, 2 * y - 1) for i, j in _modes(2, k)], axis=1)
    x, y, z = pts.T
    w, q = 1 - y - z, 1 - z
    return np.stack([math.sqrt((2 * i + 1) * (2 * i + 2 * j + 2) * (2 * i + 2 * j + 2 * l + 3.0))
                     * _jacobi(i, 0, 2 * x / w - 1) * w ** i * _jacobi(j, 2 * i + 1, 2 * y / q - 1) * q ** j
                     * _jacobi(l, 2 * i + 2 * j + 2, 2 * z - 1) for i, j, l in _modes(3, k)], axis=1)


def _grad(dim, k, pts):
    """reference gradients [q, mode, r] by the complex step"""
    return np.stack([_phi(dim, k, pts + 1e-30j * np.eye(dim)[r]).imag * 1e30 for r in range(dim)], axis=2)


def _rule(dim, n):
    """collapsed Gauss-Legendre product rule on the unit simplex"""
    g, w = np.polynomial.legendre.leggauss(n)
    g, w = (g + 1) / 2, w / 2
    if dim == 1:
        return g[:, None], w
    if dim == 2:
        a, b = (v.ravel() for v in np.meshgrid(g, g, indexing="ij"))
        return np.stack([a * (1 - b), b], axis=1), np.outer(w, w).ravel() * (1 - b)
    a, b, c = (v.ravel() for v in np.meshgrid(g, g, g, indexing="ij"))
    W = np.einsum("i,j,l->ijl", w, w, w).ravel() * (1 - b) * (1 - c) ** 2
    y = b * (1 - c)
    return np.stack([a * (1 - c - y), y, c], axis=1), W


class _Plain:
    """HDG on simplices by dense element algebra, batched over the elements."""

    def __init__(self, case, d):
        self.case, self.d = case, d
        self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        self.elastic = case["kind"] == "elastic"
        vert = d["vert"]
        dim = self.dim = vert.shape[1]
        self.elem = elem = np.sort(d["elem"].astype(np.int64), axis=1)
        self.ne = ne = elem.shape[0]
        # faces in lexicographic order of their sorted vertices, local face j opposite vertex j
        nv = vert.shape[0]
        key = np.zeros((ne, dim + 1), dtype=np.int64)
        for j in range(dim + 1):
            for a in range(dim + 1):
                if a != j:
                    key[:, j] = key[:, j] * nv + elem[:, a]
        uniq, inv, cnt = np.unique(key.ravel(), return_inverse=True, return_counts=True)
        self.ef = self.t(inv.reshape(ne, dim + 1))
        self.nf = uniq.size
        self.interior = self.t(cnt == 2)
        X = vert[elem]
        J = np.swapaxes(X[:, 1:] - X[:, :1], 1, 2)
        self.X0, self.Ji = X[:, 0], np.linalg.inv(J)
        self.detJ = self.t(np.abs(np.linalg.det(J)))
        self.Jinv = self.t(self.Ji)
        nrm = np.zeros((ne, dim + 1, dim))
        jf = np.zeros((ne, dim + 1))
        for f in range(dim + 1):
            Y = X[:, [a for a in range(dim + 1) if a != f]]
            t = Y[:, 1:] - Y[:, :1]
            v = np.stack([t[:, 0, 1], -t[:, 0, 0]], axis=1) if dim == 2 else np.cross(t[:, 0], t[:, 1])
            jf[:, f] = np.linalg.norm(v, axis=1)
            v = v / jf[:, f:f + 1]
            v *= -np.sign(np.sum(v * (X[:, f] - Y[:, 0]), axis=1))[:, None]
            nrm[:, f] = v
        self.nrm, self.jf = self.t(nrm), self.t(jf)
        # degree classes: (element ids, volume degree); the faces carry the largest degree's modes
        ks = d.get("elem_k")
        self.ks = np.full(ne, case["k"]) if ks is None else ks
        self.kt = int(self.ks.max())
        self.Nf = math.comb(self.kt + dim - 1, dim - 1)
        self.mf = self.Nf * (dim if self.elastic else 1)
        per = 1 << 27
        self.parts = []
        for kk in sorted(set(self.ks.tolist())):
            ids = np.nonzero(self.ks == kk)[0]
            n = self.n_of(kk)
            step = max(1, per // (n * n))
            self.parts += [(kk, self.t(ids[i:i + step])) for i in range(0, ids.size, step)]
        # active trace modes of every face
        kf = np.zeros(self.nf, dtype=np.int64)
        np.maximum.at(kf, inv, np.repeat(self.ks, dim + 1))
        deg = np.array([sum(i) for i in _modes(dim - 1, self.kt)])
        act = deg[None, :] <= kf[:, None]
        self.active = self.t(np.tile(act, (1, dim)) if self.elastic else act)
        self.unknown = (self.active & self.interior[:, None]).double()
        self.fact = {}

    def t(self, a):
        return torch.as_tensor(np.ascontiguousarray(a), device=self.dev)

    def n_of(self, k):
        Np = math.comb(k + self.dim, self.dim)
        return Np * (self.dim + self.dim * (self.dim + 1) // 2 if self.elastic else self.dim + 1)

    def tables(self, k):
        dim = self.dim
        q, w = _rule(dim, k + 3)
        V, G = _phi(dim, k, q), _grad(dim, k, q)
        Dr = np.einsum("q,qi,qlr->ril", w, V, G)
        e, wf = _rule(dim - 1, self.kt + 3)
        U = _phi(dim - 1, self.kt, e)
        corners = np.vstack([np.zeros(dim), np.eye(dim)])
        Fm, E = [], []
        for f in range(dim + 1):
            Y = corners[[a for a in range(dim + 1) if a != f]]
            Vf = _phi(dim, k, Y[0] + e @ (Y[1:] - Y[0]))
            Fm.append(np.einsum("q,qi,qm->im", wf, Vf, U))
            E.append(np.einsum("q,qi,ql->il", wf, Vf, Vf))
        return self.t(Dr), self.t(np.array(Fm)), self.t(np.array(E))

    def mass(self, k, ids):
        """weighted mass as (diagonal blocks [e, c, c]) over the field components"""
        d, dim = self.d, self.dim
        g = lambda a: self.t(a)[ids]
        det = self.detJ[ids]
        if not self.elastic:
            rho, c = g(d["rho"]), g(d["c"])
            return torch.diag_embed(torch.stack([det / (rho * c * c)] + [rho * det] * dim, dim=1))
        lam, mu, rho = g(d["lam"]), g(d["mu"]), g(d["rho"])
        M = torch.zeros((len(ids), 9, 9), dtype=torch.float64, device=self.dev)
        for i in range(3):
            M[:, i, i] = rho
            M[:, 3 + i, 3 + i] = 1 / (2 * mu)
            M[:, 6 + i, 6 + i] = 1 / mu
            for j in range(3):
                M[:, 3 + i, 3 + j] -= lam / ((3 * lam + 2 * mu) * 2 * mu)
        return M * det[:, None, None]

    def blocks(self, k, ids, alpha):
        """A, B, C, D of the elements `ids` (degree k)"""
        dim, Nf, mf = self.dim, self.Nf, self.mf
        Dr, Fm, E = self.tables(k)
        Np = Dr.shape[1]
        ne, det, nrm, jf = len(ids), self.detJ[ids], self.nrm[ids], self.jf[ids]
        Dx = torch.einsum("e,erj,ril->ejil", det, self.Jinv[ids], Dr)
        Es = torch.einsum("ef,fil->eil", jf, E)
        M = self.mass(k, ids)
        n = M.shape[1] * Np
        A = torch.einsum("eab,il->eaibl", alpha * M, torch.eye(Np, dtype=torch.float64, device=self.dev)).reshape(ne, n, n)
        B = torch.zeros((ne, n, (dim + 1) * mf), dtype=torch.float64, device=self.dev)
        C = torch.zeros_like(B).transpose(1, 2).contiguous()
        Dd = torch.zeros((ne, (dim + 1) * mf), dtype=torch.float64, device=self.dev)
        b = lambda a: slice(a * Np, (a + 1) * Np)
        if not self.elastic:
            A[:, b(0), b(0)] += Es
            for j in range(dim):
                A[:, b(0), b(1 + j)] += Dx[:, j]
                A[:, b(1 + j), b(0)] -= Dx[:, j].transpose(1, 2)
            for f in range(dim + 1):
                s = slice(f * Nf, (f + 1) * Nf)
                JF = jf[:, f, None, None] * Fm[f]
                B[:, b(0), s], C[:, s, b(0)] = -JF, JF.transpose(1, 2)
                for j in range(dim):
                    nj = nrm[:, f, j, None, None] * JF
                    B[:, b(1 + j), s], C[:, s, b(1 + j)] = nj, nj.transpose(1, 2)
                Dd[:, s] = -jf[:, f, None]
            return A, B, C, Dd
        rho, mu = self.t(self.d["rho"])[ids], self.t(self.d["mu"])[ids]
        st = 2.0 * rho * torch.sqrt(mu / rho)
        comps = [(0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1)]
        nE = torch.einsum("ef,efj,fil->ejil", jf, nrm, E)
        for i in range(3):
            A[:, b(i), b(i)] += st[:, None, None] * Es
        for a, (i, j) in enumerate(comps):
            for p, q in ([(i, j)] if i == j else [(i, j), (j, i)]):
                A[:, b(3 + a), b(p)] += Dx[:, q].transpose(1, 2)
                A[:, b(p), b(3 + a)] += Dx[:, q].transpose(1, 2) - nE[:, q]
                for f in range(4):
                    s = slice((f * 3 + p) * Nf, (f * 3 + p + 1) * Nf)
                    nq = nrm[:, f, q, None, None] * jf[:, f, None, None] * Fm[f]
                    B[:, b(3 + a), s] -= nq
                    C[:, s, b(3 + a)] += nq.transpose(1, 2)
        for i in range(3):
            for f in range(4):
                s = slice((f * 3 + i) * Nf, (f * 3 + i + 1) * Nf)
                JF = st[:, None, None] * jf[:, f, None, None] * Fm[f]
                B[:, b(i), s] -= JF
                C[:, s, b(i)] -= JF.transpose(1, 2)
                Dd[:, s] = (st * jf[:, f])[:, None]
        return A, B, C, Dd

    def condense(self, alpha):
        m = (self.dim + 1) * self.mf
        self.alpha, self.S = alpha, torch.empty((self.ne, m, m), dtype=torch.float64, device=self.dev)
        self.fact = []
        diag = torch.zeros((self.nf, self.mf), dtype=torch.float64, device=self.dev)
        for k, ids in self.parts:
            A, B, C, Dd = self.blocks(k, ids, alpha)
            lu, piv = torch.linalg.lu_factor(A)
            S = torch.diag_embed(Dd) - C @ torch.linalg.lu_solve(lu, piv, B)
            self.S[ids] = S
            self.fact.append((lu, piv, B, C) if self.case["kind"] != "condense" else None)
            diag.index_add_(0, self.ef[ids].reshape(-1), torch.diagonal(S, dim1=1, dim2=2).reshape(-1, self.mf))
        self.diag = torch.where(self.unknown > 0, diag, torch.ones_like(diag))

    def apply(self, x):
        """K x on the unknown trace entries; x [face, mode, column]"""
        R = x.shape[2]
        xk = (x * self.unknown[:, :, None])[self.ef].reshape(self.ne, -1, R)
        y = torch.zeros_like(x).index_add_(0, self.ef.reshape(-1), torch.bmm(self.S, xk).reshape(-1, self.mf, R))
        return y * self.unknown[:, :, None]

    def trace_solve(self, r):
        """conjugate gradients on each column of K lam = r, restarted on the true residual"""
        x = torch.zeros_like(r)
        scale = r.square().sum((0, 1)).sqrt().clamp_min(1e-300)
        for sweep in range(3):
            res = r - self.apply(x) if sweep else r * self.unknown[:, :, None]
            z = res / self.diag[:, :, None]
            p, rz, dx = z.clone(), (res * z).sum((0, 1)), torch.zeros_like(r)
            for it in range(2000):
                q = self.apply(p)
                a = rz / torch.where(rz == 0, torch.ones_like(rz), (p * q).sum((0, 1)))
                dx += a * p
                res = res - a * q
                z = res / self.diag[:, :, None]
                new = (res * z).sum((0, 1))
                if it % 8 == 7 and bool((res.square().sum((0, 1)).sqrt() <= scale * (1e-15 if sweep < 2 else 1e-17)).all()):
                    break
                if sweep and it > 60:
                    break
                p = z + torch.where(rz == 0, torch.zeros_like(rz), new / torch.where(rz == 0, torch.ones_like(rz), rz)) * p
                rz = new
            x = x + dx
        return x

    def rhs(self, F):
        """condensed right-hand side of per-part element data F (list of [e, n, R])"""
        R = F[0].shape[2]
        r = torch.zeros((self.nf, self.mf, R), dtype=torch.float64, device=self.dev)
        for (k, ids), (lu, piv, B, C), f in zip(self.parts, self.fact, F):
            g = -(C @ torch.linalg.lu_solve(lu, piv, f))
            r.index_add_(0, self.ef[ids].reshape(-1), g.reshape(-1, self.mf, R))
        return r * self.unknown[:, :, None]

    def recover(self, F, lam):
        out = []
        for (k, ids), (lu, piv, B, C), f in zip(self.parts, self.fact, F):
            lk = (lam * self.unknown[:, :, None])[self.ef[ids]].reshape(len(ids), -1, lam.shape[2])
            out.append(torch.linalg.lu_solve(lu, piv, f - B @ lk))
        return out

    def times_mass(self, u):
        out = []
        for (k, ids), v in zip(self.parts, u):
            M = self.mass(k, ids)
            out.append(torch.einsum("eab,ebir->eair", M, v.reshape(len(ids), M.shape[1], -1, v.shape[2])).reshape(v.shape))
        return out

    def source(self, t):
        """(element, modes at the point, value at time t) of each source"""
        out = []
        for x, delay in zip(self.d["src"], self.d["delay"]):
            xi = np.einsum("eij,ej->ei", self.Ji, x - self.X0)
            e = int(np.nonzero((xi.min(axis=1) >= -1e-12) & (xi.sum(axis=1) <= 1 + 1e-12))[0][0])
            a = (math.pi * F0 * (t - delay - T0)) ** 2
            out.append((e, _phi(self.dim, self.case["k"], xi[e:e + 1])[0], (1 - 2 * a) * math.exp(-a)))
        return out

    def stage(self, hist, t):
        F = [self.alpha * f for f in self.times_mass(hist)]
        if "src" in self.d:
            for col, (e, phi, val) in enumerate(self.source(t)):
                for (k, ids), f in zip(self.parts, F):
                    at = torch.nonzero(ids == e)
                    if at.numel():
                        f[int(at[0]), :phi.size, col] += val * self.t(phi)
        lam = self.trace_solve(self.rhs(F))
        return self.recover(F, lam), lam

    def initial(self):
        c, R = self.case, self.case.get("R", 1)
        u = [torch.zeros((len(ids), self.n_of(k), R), dtype=torch.float64, device=self.dev) for k, ids in self.parts]
        if self.elastic:
            for v, (k, ids) in zip(u, self.parts):
                # the L2 projection that the library's own rule of k + 2 Gauss-Jacobi points defines
                q, w = _jacobi_rule(k + 2)
                e = ids.cpu().numpy()
                X = self.d["vert"][self.elem[e]]
                x = X[:, :1] + np.einsum("qr,erj->eqj", q, X[:, 1:] - X[:, :1])
                vals = np.exp(-np.sum((x - self.d["center"]) ** 2, axis=-1) / (2 * 0.05 ** 2))
                Np = math.comb(k + 3, 3)
                v[:, 2 * Np:3 * Np, 0] = self.t(vals @ (w[:, None] * _phi(3, k, q)))
        return u

    def answer(self):
        kind, case = self.case["kind"], self.case
        lin = lambda cs, us: [sum(c * u for c, u in zip(cs, v)) for v in zip(*us)]
        if kind == "post":
            return {"p": self.post()}
        self.condense(_alpha(case))
        if kind == "condense":
            y = self.apply(self.t(self.d["x"])[:, :, None])[:, :, 0]
            return {"S": self.S, "y": y}
        if kind == "solve":
            F = [self.t(self.d["F"])[ids][:, :, None] for k, ids in self.parts]
            r = self.rhs(F)
            lam = self.trace_solve(r)
            return {"r": r[:, :, 0], "lam": lam[:, :, 0], "u": self.flat(self.recover(F, lam))}
        u = self.initial()
        dt, t = case["dt"], T_START
        if kind == "elastic":
            a, b, c = _dirk3()
            d = np.linalg.inv(a)
            e = b @ d
            for _ in range(case["steps"]):
                us = []
                for i in range(3):
                    cs = [d[i, :i + 1].sum() / d[i, i]] + [-d[i, j] / d[i, i] for j in range(i)]
                    ui, lam = self.stage(lin(cs, [u] + us), t + c[i] * dt)
                    us.append(ui)
                u = lin([1.0 - b @ d.sum(axis=1)] + list(e), [u] + us)
                t += dt
        else:
            prev = u
            for i in range(case["steps"]):
                hist = u if case["scheme"] == "be" else lin([4.0 / 3.0, -1.0 / 3.0], [u, prev])
                prev = u
                u, lam = self.stage(hist, T_START + (i + 1) * dt)
        return {"u": self.flat(u), "lam": self.flat_traces(lam)}

    def flat(self, u):
        if self.elastic and self.case["k"] == 0:
            off = np.concatenate([[0], np.cumsum([self.n_of(k) for k in self.ks])])
            out = torch.empty(int(off[-1]), dtype=torch.float64, device=self.dev)
            o = self.t(off[:-1])
            for (k, ids), v in zip(self.parts, u):
                out[(o[ids][:, None] + torch.arange(v.shape[1], device=self.dev)).reshape(-1)] = v.reshape(-1)
            return out
        out = torch.empty((self.ne,) + tuple(u[0].shape[1:]), dtype=torch.float64, device=self.dev)
        for (k, ids), v in zip(self.parts, u):
            out[ids] = v
        return out if out.shape[2] > 1 else out[:, :, 0]

    def flat_traces(self, lam):
        if self.elastic and self.case["k"] == 0:
            return lam[:, :, 0][self.active]
        return lam if lam.shape[2] > 1 else lam[:, :, 0]

    def post(self):
        """p* of degree k + 1: the mean of p and the Neumann problem with the discrete gradient"""
        dim, k = self.dim, self.case["k"]
        Dr, Fm, _ = self.tables(k)
        q, w = _rule(dim, k + 4)
        V, G1 = _phi(dim, k, q), _grad(dim, k + 1, q)
        K1 = self.t(np.einsum("q,qir,qls->rsil", w, G1, G1))
        E1 = self.t(np.einsum("q,qir,ql->ril", w, G1, V))
        u, lam = self.t(self.d["u"]), self.t(self.d["lam"])
        Np = Dr.shape[1]
        out = torch.empty((self.ne, K1.shape[2]), dtype=torch.float64, device=self.dev)
        for _, ids in self.parts:
            det, Ji = self.detJ[ids], self.Jinv[ids]
            p = u[ids][:, :Np]
            g = -torch.einsum("e,erj,ril,ei->ejl", det, Ji, Dr, p)
            for f in range(dim + 1):
                g += torch.einsum("e,ej,im,em->eji", self.jf[ids][:, f], self.nrm[ids][:, f], Fm[f], lam[self.ef[ids][:, f]])
            gr = g / det[:, None, None]
            A = torch.einsum("e,erj,esj,rsil->eil", det, Ji, Ji, K1)
            b = torch.einsum("e,erj,ril,ejl->ei", det, Ji, E1, gr)
            out[ids, 0] = p[:, 0]
            out[ids, 1:] = torch.linalg.solve(A[:, 1:, 1:], b[:, 1:])
        return out


def _jacobi_rule(n):
    """collapsed Gauss-Jacobi rule on the unit tetrahedron, n points a direction: the nodes in
    the directions of weight (1 - t)^a are the eigenvalues of the Jacobi matrix"""
    def gauss(a):
        j = np.arange(n, dtype=float)
        dia = np.where(j == 0, -a / (a + 2.0), -a * a / ((2 * j + a) * (2 * j + a + 2) + (j == 0)))
        i = np.arange(1, n, dtype=float)
        off = 2 / (2 * i + a) * np.sqrt(i * (i + a) * i * (i + a) / ((2 * i + a - 1) * (2 * i + a + 1)))
        x, v = np.linalg.eigh(np.diag(dia) + np.diag(off, 1) + np.diag(off, -1))
        return x, v[0] ** 2 * 2 ** (a + 1) / (a + 1)
    (a, wa), (b, wb), (c, wc) = gauss(0), gauss(1), gauss(2)
    A, B, C = (v.ravel() for v in np.meshgrid(a, b, c, indexing="ij"))
    z = (1 + C) / 2
    y = (1 + B) / 2 * (1 - z)
    return np.stack([(1 + A) / 2 * (1 - y - z), y, z], axis=1), np.einsum("i,j,l->ijl", wa, wb, wc).ravel() / 64

