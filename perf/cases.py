"""Performance cases: the calls of a Chebyshev-filtered subspace iteration with this library, each
through its public entry point, over the range of cells, meshes, k-points, vector counts and
arithmetic that a user runs.

A case is one call on one operator:
  "pass"        one whole iteration: build, filter, Cholesky-QR, Rayleigh-Ritz, occupations, density
  "apply"       Y = (M^O)^{-1} H^O X, the FP64-class operator application
  "filter_low"  the batched tensor-core filter of FP32 / complex64 vectors, every k-point at once
  "defect"      the batched filter in defect form (FP64 vectors, tensor-core degrees)
  "ortho"       Cholesky-QR twice in the M inner product
  "ritz"        Rayleigh-Ritz with residuals
  "density"     the density and the band-trace gradient from one evaluation of the fields
  "build"       the operator build from a new potential, and its first application
  "adjoint"     forward and backward of Y = H(V) X through autograd

The operator (mesh, enrichment, quadrature, k-points, and for the calls that do not build it, the
stored cell matrices) is the handle that a program keeps for a geometry: it is set up once and
shared by the states of a case. Potentials and vectors come from the seed.

``exact`` restates the discrete problem in plain numpy and torch, matrix free and in 64 bits.
"""
import math

import numpy as np
import torch

import paper_2010_09701_gb300 as oefe

# ------------------------------------------------------------------------------------ geometries
# name: (cell edge, nuclei in units of the edge, charges, cutoff radii r0 and rc, octree depth)
_FCC = [(0, 0, 0), (0, .5, .5), (.5, 0, .5), (.5, .5, 0)]
_ZB = _FCC + [(x + .25, y + .25, z + .25) for x, y, z in _FCC]


def _divacancy():
    sites = [((x + i) / 2, (y + j) / 2, (z + k) / 2, 14 if n < 4 else 6)
             for k in range(2) for j in range(2) for i in range(2) for n, (x, y, z) in enumerate(_ZB)]
    return [s[:3] for s in sites if s[:3] not in ((0, 0, 0), (.125, .125, .125))], \
        [s[3] for s in sites if s[:3] not in ((0, 0, 0), (.125, .125, .125))]


CELLS = {
    "tiny": (6.0, [(0, 0, 0), (.5, .5, .5)], [3, 4], 1.5, 2.5, 2),
    "2atom": (10.26, [(0, 0, 0), (.25, .25, .25)], [6, 14], 3.0, 4.0, 6),
    "8atom": (8.5, _ZB, [14] * 4 + [6] * 4, 3.0, 4.0, 6),
    "62atom": (16.4, *_divacancy(), 3.0, 4.0, 6),
}
ORBITALS = ((1, 0), (2, 0), (2, 1), (2, 2), (2, 3))     # 1s, 2s, 2p_x, 2p_y, 2p_z: (n, angular code)
KPOINTS = ((.25, .25, .25), (-.25, .25, .25), (.25, -.25, .25))   # in units of 2 pi / a
NGRID = 2000


def listed():
    """The listed cases, operators of one geometry next to each other."""
    return [
        # the smallest call: a handful of vectors on a small box, where launches and latency count
        {"name": "apply_tiny_k", "call": "apply", "cell": "tiny", "ncell": 2, "p": 3, "nk": 1, "nv": 8, "pairs": False},
        # a whole pass on the two-atom Gamma-point cell in native FP64, the library's default arithmetic
        {"name": "pass_2atom_fp64", "call": "pass", "cell": "2atom", "ncell": 8, "p": 4, "nk": 0, "nv": 20,
         "degree": 20, "pairs": False},
        # differentiating through the operator at an odd width and order (potential inversion)
        {"name": "adjoint_2atom_k_fp64", "call": "adjoint", "cell": "2atom", "ncell": 6, "p": 5, "nk": 1, "nv": 13,
         "pairs": False},
        # one FP64 filter degree / H X of the plain FP64 path with Bloch vectors
        {"name": "apply_8atom_k_fp64", "call": "apply", "cell": "8atom", "ncell": 8, "p": 6, "nk": 1, "nv": 64,
         "pairs": False},
        # the low-precision filter of all k-points in one batch
        {"name": "filter_8atom_2k_c64", "call": "filter_low", "cell": "8atom", "ncell": 8, "p": 6, "nk": 2, "nv": 64,
         "degree": 30, "pairs": True},
        # the defect-form filter at a ragged vector count per k-point
        {"name": "defect_8atom_2k", "call": "defect", "cell": "8atom", "ncell": 8, "p": 6, "nk": 2, "nv": 97,
         "degree": 30, "pairs": True},
        # projection of a block of one k-point
        {"name": "ritz_8atom_k", "call": "ritz", "cell": "8atom", "ncell": 8, "p": 6, "nk": 2, "nv": 64, "pairs": True},
        # a new potential in the self-consistency loop
        {"name": "build_8atom_2k", "call": "build", "cell": "8atom", "ncell": 8, "p": 6, "nk": 2, "nv": 16,
         "pairs": True},
        # the divacancy supercell at the Gamma point (real arithmetic, 360 vectors): the steps of one
        # pass of the large calculations, on a 16^3 mesh
        {"name": "defect_62atom_gamma", "call": "defect", "cell": "62atom", "ncell": 16, "p": 6, "nk": 0, "nv": 360,
         "degree": 50, "pairs": True},
        {"name": "ortho_62atom_gamma", "call": "ortho", "cell": "62atom", "ncell": 16, "p": 6, "nk": 0, "nv": 360,
         "pairs": True},
        {"name": "ritz_62atom_gamma", "call": "ritz", "cell": "62atom", "ncell": 16, "p": 6, "nk": 0, "nv": 360,
         "pairs": True},
        {"name": "density_62atom_gamma", "call": "density", "cell": "62atom", "ncell": 16, "p": 6, "nk": 0, "nv": 360,
         "pairs": True},
    ]


def draw(rng):
    """A case of the same ranges: any call, cells of 2 or 8 atoms, orders 3 to 6, even and odd meshes,
    1 to 128 vectors per k-point or 1 to 360 at the Gamma point, native FP64 or FP32 pairs."""
    call = rng.choice(["pass", "apply", "filter_low", "defect", "ortho", "ritz", "density", "build", "adjoint"])
    cell = rng.choice(["2atom", "8atom"])
    ncell = rng.randint(4, 9) if cell == "2atom" else rng.randint(8, 10)
    nk = rng.choice([0, 0, 1, 2, 3])
    if call == "pass":
        cell, ncell, nk = "2atom", rng.randint(4, 9), rng.choice([0, 1])
    if call in ("build", "adjoint"):
        nk, nv = min(nk, 2), rng.randint(1, 32)
    else:
        nv = int(round(math.exp(rng.uniform(0.0, math.log(360 if nk == 0 else 128)))))
    if call == "pass":
        nv = rng.randint(12, 40)
    c = {"call": call, "cell": cell, "ncell": ncell, "p": rng.randint(3, 6), "nk": nk, "nv": nv,
         "pairs": rng.random() < (0.9 if nv > 64 else 0.6)}
    if call in ("pass", "filter_low", "defect"):
        c["degree"] = rng.randint(8, 30)
    if call == "defect":
        c["pairs"] = True
    return c


# --------------------------------------------------------------------------------------- inputs
def _breakpoints(a, ncell, coords):
    """Cell boundaries of one axis: nuclear coordinates are boundaries, cells shared out by length and
    graded 1.5 to 1 toward both ends of an interval; uniform when there are too many coordinates."""
    ends = sorted({round(x % 1.0, 9) for x in coords} | {0.0})
    if len(ends) > ncell // 2:
        return np.linspace(0.0, a, ncell + 1)
    ends = np.array(ends + [1.0]) * a
    share = np.diff(ends) / a * ncell
    n = np.maximum(np.floor(share + 1e-9).astype(int), 2)
    while n.sum() > ncell:
        n[int(np.argmax(n - share))] -= 1
    while n.sum() < ncell:
        n[int(np.argmax(share - n))] += 1
    out = [0.0]
    for m, x0, x1 in zip(n, ends[:-1], ends[1:]):
        w = np.array([1.5 ** min(i, m - 1 - i) for i in range(m)])
        out += list(x0 + np.cumsum(w / w.sum()) * (x1 - x0))
    out[-1] = a
    return np.array(out)


def _radial(n, l, Z, r):
    """Hydrogenic radial function and its derivative."""
    e = np.exp(-Z * r / n)
    if n == 1:
        return 2 * Z ** 1.5 * e, -2 * Z ** 2.5 * e
    if l == 0:
        c = Z ** 1.5 / math.sqrt(8.0)
        return c * (2 - Z * r) * e, c * (-Z - Z / 2 * (2 - Z * r)) * e
    c = Z ** 2.5 / math.sqrt(24.0)
    return c * r * e, c * (1 - Z * r / 2) * e


class _Geometry:
    """The inputs that describe a cell: boundaries, nuclei, radial tables, k-points, rules."""

    def __init__(self, c):
        self.a, pos, Z, self.r0, self.rc, self.depth = CELLS[c["cell"]]
        self.pos, self.Z = np.array(pos) * self.a, np.array(Z)
        self.p, self.n = c["p"], c["ncell"]
        self.xb = [_breakpoints(self.a, self.n, [q[d] for q in pos]) for d in range(3)]
        self.nq_cell, self.nq_enr = self.p + 1, self.p + (2 if c["cell"] == "tiny" else 3)
        r = np.linspace(0.0, self.rc, NGRID)
        tab = [[_radial(n, min(m, 1), float(z), r) for n, m in ORBITALS] for z in Z]
        self.R = np.array([[t[0] for t in row] for row in tab])
        self.dR = np.array([[t[1] for t in row] for row in tab])
        self.lm = np.array([m for _, m in ORBITALS], np.int32)
        self.k = np.array(KPOINTS[:c["nk"]]).reshape(-1, 3) * 2 * math.pi / self.a if c["nk"] else np.zeros((1, 3))
        self.nh, self.nO = (self.n * self.p) ** 3, len(Z) * len(ORBITALS)

    def gll(self):
        L = np.polynomial.legendre
        co = np.eye(self.p + 1)[self.p]
        x = np.concatenate([[-1.0], np.sort(np.real(L.legroots(L.legder(co)))), [1.0]])
        return x, 2.0 / (self.p * (self.p + 1) * L.legval(x, co) ** 2)

    def axis_nodes(self, d):
        """Coordinates of the distinct nodes of an axis."""
        x, _ = self.gll()
        b = self.xb[d]
        return np.concatenate([b[i] + (x[:-1] + 1) / 2 * (b[i + 1] - b[i]) for i in range(self.n)])

    def potential(self, pts):
        """Gaussian-smeared nuclear Coulomb potential on the minimal image."""
        V = torch.zeros(pts.shape[0], dtype=torch.float64, device=pts.device)
        for R, z in zip(self.pos, self.Z):
            d = pts - torch.as_tensor(R, device=pts.device)
            r = torch.linalg.vector_norm(d - self.a * torch.round(d / self.a), dim=1).clamp_min(1e-9)
            V -= float(z) * torch.special.erf(r / (math.sqrt(2.0) * 0.05)) / r
        return V

    def ripple(self, pts, seed):
        """A smooth change of the potential, another for each seed (the density of the last pass)."""
        g = np.random.default_rng(seed)
        V = torch.zeros(pts.shape[0], dtype=torch.float64, device=pts.device)
        for _ in range(4):
            m = torch.as_tensor(g.integers(-2, 3, 3) * 2 * math.pi / self.a, dtype=torch.float64, device=pts.device)
            V += 0.3 * g.uniform(0.5, 1.0) * torch.cos(pts @ m + g.uniform(0, 2 * math.pi))
        return V

    def waves(self, nv, cplx, seed, noise=1e-2):
        """A block of low-energy vectors: distinct plane waves at the nodes with a little noise, and
        random enrichment coefficients (rows: nodes x fastest, then enrichment functions)."""
        dev = _device()
        gen = torch.Generator(device=dev).manual_seed(seed)
        u = lambda *s: torch.rand(*s, generator=gen, device=dev, dtype=torch.float64) * 2 - 1  # noqa: E731
        q = np.arange(-6, 7)
        M = np.stack(np.meshgrid(q, q, q, indexing="ij"), -1).reshape(-1, 3)
        if not cplx:   # one of each pair (m, -m), a random phase makes it sine or cosine
            M = M[(M[:, 2] > 0) | ((M[:, 2] == 0) & ((M[:, 1] > 0) | ((M[:, 1] == 0) & (M[:, 0] >= 0))))]
        M = M[np.lexsort((M[:, 0], M[:, 1], M[:, 2], (M * M).sum(1)))][:nv]
        ph = u(nv) * (0.7 if not cplx else math.pi)
        dt = torch.complex128 if cplx else torch.float64
        E = []
        for d in range(3):
            x = torch.as_tensor(self.axis_nodes(d), device=dev) * (2 * math.pi / self.a)
            E.append(torch.exp(1j * x[:, None] * torch.as_tensor(M[:, d], device=dev)[None, :]))
        E[0] = E[0] * torch.exp(1j * ph)
        X = torch.empty(self.nh + self.nO, nv, dtype=dt, device=dev)
        N = self.n * self.p
        for z in range(N):   # one plane of nodes at a time
            pl = (E[0][None, :, :] * E[1][:, None, :] * E[2][z]).reshape(N * N, nv)
            nz = noise * u(N * N, nv) if not cplx else noise * torch.complex(u(N * N, nv), u(N * N, nv))
            X[z * N * N:(z + 1) * N * N] = (pl if cplx else pl.real) + nz
        xo = 0.3 * u(self.nO, nv)
        X[self.nh:] = torch.complex(xo, 0.3 * u(self.nO, nv)) if cplx else xo
        return X


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


# the operator handle of the case at hand (one is kept, as a program keeps it for its geometry)
_kept = {}


def _operator(c):
    builds = c["call"] in ("pass", "build", "adjoint")
    key = (c["cell"], c["ncell"], c["p"], c["nk"], c["pairs"], builds)
    if key not in _kept:
        for old in list(_kept):
            _kept.pop(old)[0].close()
        G = _Geometry(c)
        ctx = oefe.Context(0)
        ctx.mesh(G.a, G.xb, G.p)
        ctx.enrichment(G.pos, G.lm, G.R, G.dR, G.r0, G.rc)
        ctx.quadrature(G.nq_cell, G.nq_enr, G.depth)
        ctx.kpoints(G.k, np.full(len(G.k), 1.0 / len(G.k)))
        pts = torch.as_tensor(ctx.quadrature_points()[0], device="cuda")
        V = G.potential(pts)
        store = oefe.STORE_F64 | oefe.STORE_BF16X3
        if c["pairs"]:
            store |= oefe.STORE_F64PAIR
            ctx.set_f64_products(oefe.F64_PAIRS)
            if c["nk"] == 0:
                store |= oefe.STORE_COMPACT   # how the large Gamma-point cells are stored
        ctx.build_hamiltonian(V, store)
        if c["nk"] == 0:
            ctx.set_filter_shape(5)           # 128-vector tiles, the shape that tuning keeps for real data
        v0 = G.waves(1, c["nk"] > 0, 1, noise=1.0)
        top = max(ctx.upper_bound(k, v0, 20) for k in range(len(G.k)))
        ctx.release_workspace()
        _kept[key] = (ctx, G, pts if builds else None, V, store, _round_up(top))
    return _kept[key]


def _round_up(x):
    """The filter's upper bound, a round number above the Lanczos bound."""
    s = 10.0 ** (math.floor(math.log10(x)) - 1)
    return math.ceil(1.03 * x / s) * s


def _occ(nv):
    return 2.0 * np.linspace(1.0, 0.0, nv) ** 2


def _window(G):
    """Lower end of the filtered interval, lowest wanted value."""
    return 2.0, -0.5 * float(G.Z.max()) ** 2 - 4.0


def prepare(case, seed):
    ctx, G, pts, V, store, top = _operator(case)
    call, nv, cplx, nk = case["call"], case["nv"], case["nk"] > 0, len(G.k)
    lo, low = _window(G)
    s = {"call": call, "ctx": ctx, "store": store, "bounds": (lo, top, low), "degree": case.get("degree", 0), "nv": nv,
         "electrons": min(float(G.Z.sum()), 1.5 * nv), "w": np.full(nk, 1.0 / nk)}
    one = call in ("apply", "ortho", "ritz", "adjoint", "pass", "build")   # blocks of the first k-point only
    X = [G.waves(nv, cplx, 1000 * seed + k) for k in range(1 if one else nk)]
    if call == "ortho":   # columns as a filter leaves them: scaled by its gain at their energies
        X[0] *= torch.logspace(0, -3, nv, dtype=torch.float64, device="cuda")
    if call == "filter_low":
        X = [x.to(torch.complex64 if cplx else torch.float32) for x in X]
    if pts is not None:
        s["V"] = V + G.ripple(pts, seed)
    if call == "defect":   # values of the vectors the block approximates
        s["theta"] = [np.linspace(0.5 * low, lo, nv) for _ in range(nk)]
    s["X0"] = X
    s["X"] = [torch.empty_like(x) for x in X]
    if call == "adjoint":
        s["X0"] = [X[0].requires_grad_(True)]
        s["G"] = G.waves(nv, cplx, 1000 * seed + 500)
    if call in ("pass", "density"):
        s["rho"] = torch.empty(ctx.quadrature_count(), dtype=torch.float64, device="cuda")
        s["gV"] = torch.empty_like(s["rho"])
        s["occ"] = [_occ(nv) for _ in range(nk)]
    return s


def run(s):
    call, ctx, X, X0 = s["call"], s["ctx"], s["X"], s["X0"]
    lo, top, low = s["bounds"]
    if call == "apply":
        return ctx.apply_a(0, X0[0], X[0])
    if call == "density":
        return list(ctx.density_grad(X0, s["occ"], s["rho"], 0, s["gV"]))
    if call == "adjoint":
        from paper_2010_09701_gb300.autograd import apply_h
        V, x = s["V"].clone().requires_grad_(True), X0[0].detach().requires_grad_(True)
        Y = apply_h(V, x, ctx, 0)
        Y.backward(s["G"])
        return [Y.detach(), V.grad, x.grad]
    if call == "build":
        ctx.build_hamiltonian(s["V"], s["store"])
        return ctx.apply_h(0, X0[0], X[0])
    if call == "pass":
        ctx.build_hamiltonian(s["V"], s["store"])
    for x, x0 in zip(X, X0):
        x.copy_(x0)
    if call == "filter_low":
        return ctx.filter_batched(X, s["degree"], lo, top, low, oefe.FILTER_BF16X3)
    if call == "defect":
        return ctx.filter_batched_defect(X, s["degree"], lo, top, low, s["theta"], oefe.FILTER_BF16X3)
    if call == "ortho":
        return [X[0], ctx.orthonormalize(0, X[0])]
    if call == "ritz":
        eig, res = ctx.rayleigh_ritz(0, X[0], resid=True)
        return [eig, res, X[0]]
    ctx.chebyshev_filter(0, X[0], s["degree"], lo, top, low)   # call == "pass", one k-point
    ctx.orthonormalize(0, X[0])
    eig = ctx.rayleigh_ritz(0, X[0])
    mu, occ, band = oefe.occupations([eig], s["w"], s["electrons"])
    ctx.density_grad([X[0]], occ, s["rho"], 0, s["gV"])
    return [eig, band, s["rho"], s["gV"], X[0]]


# ----------------------------------------------------------------------------------------- work
def _cells(G):
    """Per cell: 0 plain, 1 meets an enrichment ball, 2 holds a nucleus; and its active functions."""
    img = G.pos[None, :, :] + np.array([-1, 0, 1])[:, None, None] * G.a            # (3, atoms, 3)
    best = []
    for d in range(3):
        lo, hi = G.xb[d][:-1, None, None], G.xb[d][1:, None, None]
        y = img[None, :, :, d]
        best.append(np.maximum(np.maximum(lo - y, y - hi), 0.0).min(1))             # (cells of the axis, atoms)
    x, y, z = best
    d2 = z[:, None, None] ** 2 + y[None, :, None] ** 2 + x[None, None, :] ** 2      # (z, y, x, atoms)
    t = 1e-12 * G.a
    holds = (z <= t)[:, None, None] & (y <= t)[None, :, None] & (x <= t)[None, None, :]
    near = d2 < G.rc ** 2
    act = near.copy()
    for ax in range(3):
        act = act | np.roll(act, 1, ax) | np.roll(act, -1, ax)
    cls = np.where(holds.any(-1), 2, np.where(near.any(-1), 1, 0))
    return cls.reshape(-1), act.sum(-1).reshape(-1) * len(ORBITALS), holds.reshape(-1, len(G.Z))


def work(case):
    """Bytes: inputs once and outputs once, with the stored operator read where the call applies it.
    Operations: products by sum factorization on cells with one rule, dense on the refined ones."""
    G = _Geometry(case)
    cls, ne, _ = _cells(G)
    call, nv, nk = case["call"], case["nv"], len(G.k)
    R = 2 if case["nk"] else 1
    P, n = G.p + 1, float(G.nh + G.nO)
    n1 = np.where(cls == 0, G.nq_cell, G.nq_enr).astype(float)
    naug, ne = P ** 3 + ne.astype(float), ne.astype(float)
    leaves = np.where(cls == 2, 7 * G.depth + 1, 1)
    nq = float((leaves * n1 ** 3).sum())
    to_pts = P * P * n1 * P + P * n1 * n1 * P + n1 ** 3 * P
    kin = 20 * P ** 4 if R == 2 else 7 * P ** 4
    cc = np.where(cls == 2, 0.0, R * 2 * to_pts + kin)
    enr = R * R * np.where(cls == 2, naug ** 2, P ** 3 * ne + ne * naug)
    prod = 2 * float((cc + enr).sum()) * nv                              # one FP64-class product of nv vectors
    strips = 8 * R * float(np.where(cls == 2, naug ** 2, P ** 3 * ne + ne * naug).sum())
    dense = 2.0 * float((naug ** 2).sum()) * R * R * nv                  # one tensor-core degree
    split = 4 * R * float((naug ** 2).sum())
    fields = 2 * float((leaves * (R * to_pts + n1 ** 3 * (R * R * ne + 2 * R))).sum()) * nv
    vec = 8 * R * n * nv
    PS = P * (P + 1) / 2
    build = 2 * float((leaves * (n1 * n1 * PS * n1 + n1 * PS * PS * n1 + P ** 6 / 2 * n1 + R * R * n1 ** 3 * ne * (ne + 1) / 2 +
                                 R * ne * to_pts)).sum())
    gram = 2 * R * R * n * nv * nv
    table = 8 * R * float((leaves * n1 ** 3 * ne).sum())                 # enrichment values at the points
    if call == "apply":
        return {"bytes": 2 * vec + strips, "flops": prod}
    if call == "filter_low":
        return {"bytes": nk * (vec + split), "flops": nk * case["degree"] * dense}
    if call == "defect":
        return {"bytes": nk * (2 * vec + strips + split), "flops": nk * (prod + case["degree"] * dense)}
    if call == "ortho":
        return {"bytes": 2 * vec, "flops": 2 * gram}
    if call == "ritz":
        return {"bytes": 2 * vec + strips, "flops": prod + 2.5 * gram}
    if call == "density":
        return {"bytes": nk * (vec + table) + 16 * nq, "flops": nk * fields}
    if call == "build":
        return {"bytes": 8 * nq + nk * (table + strips + split) + 2 * vec, "flops": nk * build + prod}
    if call == "adjoint":
        return {"bytes": 16 * nq + nk * table + strips + 4 * vec, "flops": nk * build + 2 * prod + 2 * fields}
    return {"bytes": 24 * nq + 2 * table + strips + 2 * vec,
            "flops": build + (case["degree"] + 1) * prod + 3 * gram + fields}


# ---------------------------------------------------------------------------------------- exact
class _Problem:
    """The discrete problem of one k-point, matrix free: fields of a block at the quadrature points
    by 1D interpolation per box plus the enrichment functions evaluated there, and the adjoint."""

    def __init__(self, G, k):
        self.G, self.k, self.dev = G, np.asarray(k), _device()
        self.cplx = bool(np.any(k))
        self.dt = torch.complex128 if self.cplx else torch.float64
        T = lambda x: torch.as_tensor(np.ascontiguousarray(x), device=self.dev)  # noqa: E731
        xn, wn = G.gll()
        h = [np.diff(b) for b in G.xb]
        m1 = []
        for d in range(3):
            m = np.zeros(G.n * G.p)
            for i in range(G.n):
                np.add.at(m, (i * G.p + np.arange(G.p + 1)) % len(m), wn * h[d][i] / 2)
            m1.append(m)
        self.m = T((m1[2][:, None, None] * m1[1][None, :, None] * m1[0][None, None, :]).reshape(-1))
        # boxes of the quadrature in the library's order
        cls, _, holds = _cells(G)
        boxes, n1s = [], []
        for e in range(G.n ** 3):
            i = (e % G.n, (e // G.n) % G.n, e // G.n ** 2)
            lo = np.array([G.xb[d][i[d]] for d in range(3)])
            hi = np.array([G.xb[d][i[d] + 1] for d in range(3)])
            lv = self._split(lo, hi, G.pos[holds[e]], 0) if cls[e] == 2 else [(lo, hi)]
            boxes += [(e, *b) for b in lv]
            n1s += [G.nq_cell if cls[e] == 0 else G.nq_enr] * len(lv)
        q0 = np.concatenate([[0], np.cumsum(np.array(n1s) ** 3)])
        self.nq = int(q0[-1])
        self.w = torch.empty(self.nq, dtype=torch.float64, device=self.dev)
        self.pts = torch.empty(self.nq, 3, dtype=torch.float64, device=self.dev)
        r = np.arange(G.p + 1)
        self.chunks = []
        for n1 in sorted(set(n1s)):
            ids = [b for b in range(len(boxes)) if n1s[b] == n1]
            t, tw = np.polynomial.legendre.leggauss(n1)
            for c0 in range(0, len(ids), 128):
                bx = ids[c0:c0 + 128]
                e = np.array([boxes[b][0] for b in bx])
                lo, hi = np.array([boxes[b][1] for b in bx]), np.array([boxes[b][2] for b in bx])
                ci = np.stack([e % G.n, (e // G.n) % G.n, e // G.n ** 2], 1)
                L, D, x, wq = [], [], [], []
                for d in range(3):
                    xd = lo[:, d, None] + (t + 1) / 2 * (hi - lo)[:, d, None]
                    hc = h[d][ci[:, d]][:, None]
                    v, dv = self._lagrange(xn, 2 * (xd - G.xb[d][ci[:, d]][:, None]) / hc - 1)
                    L.append(T(v))
                    D.append(T(dv * (2 / hc)[..., None]))
                    x.append(xd)
                    wq.append(tw * (hi - lo)[:, d, None] / 2)
                g = [(ci[:, d, None] * G.p + r) % (G.n * G.p) for d in range(3)]
                N = G.n * G.p
                nodes = g[0][:, None, None, :] + N * (g[1][:, None, :, None] + N * g[2][:, :, None, None])
                q = T((q0[bx][:, None] + np.arange(n1 ** 3)).reshape(-1))
                one = np.ones((len(bx), n1, n1, n1))
                self.pts[q] = T(np.stack([x[0][:, None, None, :] * one, x[1][:, None, :, None] * one,
                                          x[2][:, :, None, None] * one], -1).reshape(-1, 3))
                self.w[q] = T((wq[0][:, None, None, :] * wq[1][:, None, :, None] * wq[2][:, :, None, None]).reshape(-1))
                mid, half = (lo + hi) / 2, (hi - lo) / 2
                dd = np.abs(mid[:, None] - G.pos - G.a * np.round((mid[:, None] - G.pos) / G.a)) - half[:, None]
                atoms = np.where((np.maximum(dd, 0) ** 2).sum(-1).min(0) < G.rc ** 2)[0]
                self.chunks.append((n1, T(nodes.reshape(-1)), q, L, D, atoms))
        # orthogonalizing coefficients c (Eq. orthCGLL) and the enrichment overlap block
        self.c = torch.zeros(G.nO, G.nh, dtype=self.dt, device=self.dev)
        maa = torch.zeros(G.nO, G.nO, dtype=self.dt, device=self.dev)
        d = torch.zeros(G.nh, G.nO, dtype=self.dt, device=self.dev)
        for ch in self.chunks:
            f, A, _ = self._enrichment(ch, False)
            if len(f) == 0:
                continue
            wA = self.w[ch[2]][:, None] * A
            maa[f[:, None], f[None, :]] += A.conj().T @ wA
            d.index_put_((ch[1][:, None], f[None, :]), self._back(ch, wA, None), accumulate=True)
        self.c = (d / self.m[:, None]).T.contiguous()
        moo = maa - (self.c.conj() * self.m) @ self.c.T
        self.moo = (moo + moo.conj().T) / 2

    def _split(self, lo, hi, pos, level):
        G, t = self.G, 1e-12 * self.G.a
        y = pos[None] + np.array([-1, 0, 1])[:, None, None] * G.a
        if level < G.depth and ((lo - t <= y) & (y <= hi + t)).any(0).all(-1).any():
            m, out = (lo + hi) / 2, []
            for c in range(8):
                b = np.array([c & 1, (c >> 1) & 1, c >> 2], bool)
                out += self._split(np.where(b, m, lo), np.where(b, hi, m), pos, level + 1)
            return out
        return [(lo, hi)]

    @staticmethod
    def _lagrange(xn, x):
        P = len(xn)
        v, dv = np.ones(x.shape + (P,)), np.zeros(x.shape + (P,))
        for a in range(P):
            for b in range(P):
                if b != a:
                    v[..., a] *= (x - xn[b]) / (xn[a] - xn[b])
            for c in range(P):
                if c != a:
                    t = np.full(x.shape, 1.0 / (xn[a] - xn[c]))
                    for b in range(P):
                        if b not in (a, c):
                            t *= (x - xn[b]) / (xn[a] - xn[b])
                    dv[..., a] += t
        return v, dv

    def _enrichment(self, ch, grad):
        """Indices, values and gradients of the enrichment functions that reach a chunk's points."""
        G, x = self.G, self.pts[ch[2]]
        nf = len(ORBITALS)
        f = torch.as_tensor([I * nf + j for I in ch[5] for j in range(nf)], dtype=torch.int64, device=self.dev)
        A = torch.zeros(len(x), len(f), dtype=self.dt, device=self.dev)
        D = [torch.zeros_like(A) for _ in range(3)] if grad else None
        k = torch.as_tensor(self.k, device=self.dev)
        dr = G.rc / (NGRID - 1)
        for n, I in enumerate(ch[5]):
            d = x - torch.as_tensor(G.pos[I], device=self.dev)
            d = d - G.a * torch.round(d / G.a)
            r = torch.linalg.vector_norm(d, dim=1)
            inside = r < G.rc
            rs = torch.where(inside, r, torch.zeros_like(r)) / dr
            i = rs.floor().long().clamp_max(NGRID - 2)
            t = rs - i
            s = (G.rc - r) / (G.rc - G.r0)
            ex = lambda y: torch.where(y > 0, torch.exp(-1 / y.clamp_min(1e-300)), torch.zeros_like(y))  # noqa: E731
            dx = lambda y: torch.where(y > 0, ex(y) / y.clamp_min(1e-150) ** 2, torch.zeros_like(y))     # noqa: E731
            a, b = ex(s), ex(1 - s)
            h = a / (a + b)
            dh = -(dx(s) * b + a * dx(1 - s)) / (a + b) ** 2 / (G.rc - G.r0)
            r1 = r.clamp_min(1e-300)
            ph = torch.exp(-1j * (d @ k)) if self.cplx else torch.ones_like(r)
            for j in range(nf):
                R, dR = (torch.as_tensor(tb[I, j], device=self.dev) for tb in (G.R, G.dR))
                v = ((2 * t ** 3 - 3 * t ** 2 + 1) * R[i] + (t ** 3 - 2 * t ** 2 + t) * dr * dR[i] +
                     (3 * t ** 2 - 2 * t ** 3) * R[i + 1] + (t ** 3 - t ** 2) * dr * dR[i + 1])
                dv = ((6 * t ** 2 - 6 * t) * R[i] + (3 * t ** 2 - 4 * t + 1) * dr * dR[i] +
                      (6 * t - 6 * t ** 2) * R[i + 1] + (3 * t ** 2 - 2 * t) * dr * dR[i + 1]) / dr
                g, dg = torch.where(inside, v * h, 0 * r), torch.where(inside, dv * h + v * dh, 0 * r)
                code = int(G.lm[j])
                if code == 0:
                    val, gr = g / math.sqrt(4 * math.pi), [dg / r1 * d[:, e] / math.sqrt(4 * math.pi) for e in range(3)]
                else:
                    y = math.sqrt(3 / (4 * math.pi))
                    val = y * d[:, code - 1] * g / r1
                    gr = [y * d[:, code - 1] * (dg - g / r1) / r1 * d[:, e] / r1 + (y * g / r1 if e == code - 1 else 0)
                          for e in range(3)]
                A[:, n * nf + j] = ph * val
                if grad:
                    for e in range(3):
                        D[e][:, n * nf + j] = ph * (gr[e] - 1j * float(self.k[e]) * val if self.cplx else gr[e])
        return f, A, D

    def _contract(self, T, L):
        """(box, z, y, x, column) through one matrix per axis, x first."""
        for d in range(3):
            T = torch.einsum("bqa,%s->%s" % (("bzyaj", "bzyqj"), ("bzaxj", "bzqxj"), ("bayxj", "bqyxj"))[d],
                             L[d].to(T.dtype), T)
        return T

    def _points(self, ch, x, grad):
        """Values (and gradients) at a chunk's points of CFE columns x (nodes of the chunk)."""
        _, _, _, L, D, _ = ch
        B, P = L[0].shape[0], self.G.p + 1
        x = x.reshape(B, P, P, P, -1)
        flat = lambda y: y.reshape(-1, y.shape[-1])  # noqa: E731
        u = flat(self._contract(x, L))
        if not grad:
            return u, None
        return u, [flat(self._contract(x, [D[e] if e == d else L[e] for e in range(3)])) for d in range(3)]

    def _back(self, ch, s, fl):
        """The adjoint: sums of values s and fluxes fl against the CFE functions, per box and node."""
        n1, _, _, L, D, _ = ch
        B = L[0].shape[0]
        Lt, Dt = [x.transpose(1, 2) for x in L], [x.transpose(1, 2) for x in D]
        sh = lambda y: y.reshape(B, n1, n1, n1, -1)  # noqa: E731
        out = self._contract(sh(s), Lt)
        if fl is not None:
            for d in range(3):
                out = out + self._contract(sh(fl[d]), [Dt[e] if e == d else Lt[e] for e in range(3)])
        return out.reshape(-1, s.shape[-1])

    def _efe(self, X):
        nh = self.G.nh
        return X[:nh] - self.c.T @ X[nh:], X[nh:]

    def fields(self, X):
        """u at every point (columns of X)."""
        xc, xo = self._efe(X)
        u = torch.empty(self.nq, X.shape[1], dtype=self.dt, device=self.dev)
        for ch in self.chunks:
            f, A, _ = self._enrichment(ch, False)
            u[ch[2]] = self._points(ch, xc[ch[1]], False)[0] + A @ xo[f]
        return u

    def point_sums(self, X, occ, Y=None):
        """sum_v occ |u_v|^2 and Re sum_v conj(u_Y,v) u_X,v (Y = X when not given) at every point."""
        xc, xo = self._efe(X)
        yc, yo = (xc, xo) if Y is None else self._efe(Y)
        out = torch.empty(2, self.nq, dtype=torch.float64, device=self.dev)
        for ch in self.chunks:
            f, A, _ = self._enrichment(ch, False)
            u = self._points(ch, xc[ch[1]], False)[0] + A @ xo[f]
            g = u if Y is None else self._points(ch, yc[ch[1]], False)[0] + A @ yo[f]
            if occ is not None:
                out[0, ch[2]] = (u.abs() ** 2) @ occ
            out[1, ch[2]] = (g.conj() * u).real.sum(1)
        return out

    def H(self, V, X):
        G = self.G
        xc, xo = self._efe(X)
        yc, yo = torch.zeros_like(xc), torch.zeros_like(xo)
        kk = float(self.k @ self.k) / 2
        for ch in self.chunks:
            f, A, D = self._enrichment(ch, True)
            u, du = self._points(ch, xc[ch[1]], True)
            u = u + A @ xo[f]
            du = [du[e] + D[e] @ xo[f] for e in range(3)]
            w = self.w[ch[2]][:, None]
            s = w * (V[ch[2]][:, None] + kk) * u
            fl = [w * du[e] / 2 for e in range(3)]
            if self.cplx:
                for e in range(3):
                    s = s - 0.5j * float(self.k[e]) * w * du[e]
                    fl[e] = fl[e] + 0.5j * float(self.k[e]) * w * u
            yc.index_add_(0, ch[1], self._back(ch, s, fl))
            yo[f] += A.conj().T @ s + sum(D[e].conj().T @ fl[e] for e in range(3))
        return torch.cat([yc, yo - self.c.conj() @ yc])

    def M(self, X):
        return torch.cat([self.m[:, None] * X[:self.G.nh], self.moo @ X[self.G.nh:]])

    def Minv(self, Y):
        return torch.cat([Y[:self.G.nh] / self.m[:, None], torch.linalg.solve(self.moo, Y[self.G.nh:])])

    def filter(self, V, X, degree, a, b, a0):
        """The scaled three-term recurrence of the Chebyshev filter."""
        e, c = (b - a) / 2, (b + a) / 2
        s1 = s = e / (a0 - c)
        A = lambda Y: self.Minv(self.H(V, Y)) - c * Y  # noqa: E731
        prev, cur = X, s1 / e * A(X)
        for _ in range(2, degree + 1):
            s2 = 1 / (2 / s1 - s)
            prev, cur, s = cur, 2 * s2 / e * A(cur) - s * s2 * prev, s2
        return cur

    def ritz(self, V, X):
        """Ritz values, vectors and residuals of the block X."""
        HX, MX = self.H(V, X), self.M(X)
        S = MX.conj().T @ X
        Li = torch.linalg.inv(torch.linalg.cholesky((S + S.conj().T) / 2))
        h = X.conj().T @ HX
        eig, U = torch.linalg.eigh(Li @ ((h + h.conj().T) / 2) @ Li.conj().T)
        U = Li.conj().T @ U
        Rs = HX @ U - (MX @ U) * eig
        num = (Rs.conj() * self.Minv(Rs)).real.sum(0).clamp_min(0).sqrt()
        return eig, num, X @ U


def exact(case, seed):
    """What run returns, in 64 bits; None where the matrix-free problem takes too long here, and in
    the place of vectors that are determined up to a phase only."""
    G = _Geometry(case)
    call, nv, cplx, nk = case["call"], case["nv"], case["nk"] > 0, len(G.k)
    apps = {"pass": case.get("degree", 0) + 2, "filter_low": case.get("degree", 0),
            "defect": case.get("degree", 0)}.get(call, 1)
    cls, ne, _ = _cells(G)   # work of an application, in multiplications per vector
    leaves = np.where(cls == 2, 7 * G.depth + 1, 1)
    per = float((leaves * (G.p + 4) ** 3 * (ne + 8 * (G.p + 1))).sum()) * (4 if cplx else 1)
    apps *= {"density": 1, "ortho": 0}.get(call, 8)
    if apps * nv * nk * per > 1e13 or (case["cell"] == "62atom" and call != "ortho"):
        return None
    lo, low = _window(G)
    P = [_Problem(G, k) for k in G.k]
    V = G.potential(P[0].pts)
    one = call in ("apply", "ortho", "ritz", "adjoint", "pass", "build")
    X = [G.waves(nv, cplx, 1000 * seed + k) for k in range(1 if one else nk)]
    if call in ("pass", "build", "adjoint"):
        V0, V = V, V + G.ripple(P[0].pts, seed)
    if call == "apply":
        return P[0].Minv(P[0].H(V, X[0]))
    if call == "build":
        return P[0].H(V, X[0])
    if call == "ritz":
        eig, res, _ = P[0].ritz(V, X[0])
        return [eig, res, None]
    if call == "ortho":
        x = X[0] * torch.logspace(0, -3, nv, dtype=torch.float64, device=_device())
        S = P[0].M(x).conj().T @ x
        S = (S + S.conj().T) / 2
        sc = torch.exp2(-(torch.frexp(S.diagonal().real.sqrt())[1].double()))
        L = torch.linalg.cholesky(sc[:, None] * S * sc)
        l = L.diagonal().real
        q = torch.linalg.solve_triangular(L.conj(), (x * sc).T, upper=False).T
        return [q, float((l.max() / l.min()) ** 2)]
    if call == "adjoint":
        g = G.waves(nv, cplx, 1000 * seed + 500)
        return [P[0].H(V, X[0]), P[0].w * P[0].point_sums(X[0], None, g)[1], P[0].H(V, g)]
    if call == "density":
        occ = torch.as_tensor(_occ(nv), device=_device())
        sums = [p.point_sums(x, occ) for p, x in zip(P, X)]
        return [sum(s[0] for s in sums), P[0].w * sums[0][1]]
    top = _operator(case)[5]   # the bound is an input of the call
    if call in ("filter_low", "defect"):
        X = [x.to(torch.complex64 if cplx else torch.float32).to(p.dt) if call == "filter_low" else x
             for x, p in zip(X, P)]
        return [p.filter(V, x, case["degree"], lo, top, low) for p, x in zip(P, X)]
    eig, _, x = P[0].ritz(V, P[0].filter(V, X[0], case["degree"], lo, top, low))
    e = eig.cpu().numpy()
    ne, kT = min(float(G.Z.sum()), 1.5 * nv), 3.166811563e-6 * 500.0
    fd = lambda mu: 1 / (1 + np.exp(np.clip((e - mu) / kT, -700, 700)))  # noqa: E731
    a, b = e.min() - 1, e.max() + 1
    for _ in range(200):
        a, b = ((a + b) / 2, b) if 2 * fd((a + b) / 2).sum() < ne else (a, (a + b) / 2)
    f = 2 * fd((a + b) / 2)
    s = P[0].point_sums(x, torch.as_tensor(f, device=_device()))
    return [eig, float((f * e).sum()), s[0], P[0].w * s[1], None]
