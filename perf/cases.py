"""Timed cases: what a user of the solver has it do on one GPU, through the public calls of
paper_1605_04521_gb300.oras.

Every problem is the unit cube split into n^3 cubes of 6 tetrahedra (Kuhn), filled with the gel of
the imaging chamber (eps_r = 44 - 20i) and a head-like ball with a small inclusion whose radius and
permittivity come from the seed, as the serving stream draws them.  Sources are point dipoles near
the antenna ring, turned by the seed.

Solves run to 1e-11, so that the returned field is fixed far below the digits that the rounding of a
preconditioner (which only steers the iteration) can move.
"""
import itertools
import math

import numpy as np
import torch

from paper_1605_04521_gb300 import oras as O

EPS_GEL = complex(44.0, -20.0)
K0 = 2.0 * math.pi * 2.0 / np.sqrt(EPS_GEL).real      # two in-medium wavelengths across the cube
TOL = 1e-11
NNZ_ROW = {1: 15.5, 2: 42.0, 3: 81.0}                 # nonzeros a row of A, roughly


def listed():
    return [
        # the benchmark: one imaging-loop step (new permittivities: assembly, local
        # factorisations, solve) of the 16^3 degree-2 head problem, at its tuned panel width
        dict(name="step_head16", kind="step", n=16, r=2, nsub=64, overlap=2, k=1, bits=32, restart=100, panel=192),
        # the same step on the 8^3 profiling problem, default options
        dict(name="step_head8", kind="step", n=8, r=2, nsub=8, overlap=1, k=1, bits=32, restart=50, panel=0),
        # the smallest step (the parity-test size): latency and launches
        dict(name="step_small4", kind="step", n=4, r=2, nsub=8, overlap=1, k=1, bits=32, restart=50, panel=0),
        # degree 3 with 8 dipoles, as the serving stream sends it; 9^3 cubes, ragged subdomains
        dict(name="step_deg3_k8", kind="step", n=9, r=3, nsub=32, overlap=1, k=8, bits=32, restart=50, panel=0),
        # FP64 local factors, degree 1: the double-precision configuration
        dict(name="step_cube8_fp64", kind="step", n=8, r=1, nsub=8, overlap=1, k=1, bits=64, restart=50, panel=0),
        # a long one-antenna solve with kept factors: many subdomains, no overlap, restarts
        dict(name="solve_krylov24", kind="solve", n=24, r=2, nsub=512, overlap=0, k=1, bits=32, restart=50, panel=0),
        # the 32 antennas of a ring solved together with kept factors
        dict(name="solve_ring32", kind="solve", n=16, r=2, nsub=128, overlap=1, k=32, bits=32, restart=100, panel=0),
        # three antennas together, degree 3 without overlap: the small grouped passes
        dict(name="solve_deg3_k3", kind="solve", n=10, r=3, nsub=64, overlap=0, k=3, bits=32, restart=100, panel=0),
        # the chamber with waveguide ports: new materials, the port loads solved together, S matrix
        dict(name="chamber_ports", kind="chamber", n=10, r=2, nsub=16, overlap=1, k=8, bits=32, restart=50, panel=0),
        # one request from host data to host field: set-up, load, solve, clean-up
        dict(name="request_host", kind="request", n=7, r=2, nsub=8, overlap=1, k=2, bits=32, restart=50, panel=0),
        # products with A outside a solve: residuals of 8 fields (FP64) ...
        dict(name="matvec_f64_k8", kind="matvec", n=20, r=2, nsub=256, overlap=0, k=8, bits=32, restart=50, panel=0),
        # ... and of one FP32-valued field, degree 3
        dict(name="matvec_c64_deg3", kind="matvec_c64", n=12, r=3, nsub=128, overlap=0, k=1, bits=32, restart=50, panel=0),
    ]


def draw(rng):
    """Problems between the smallest and the largest listed ones, subdomains of the serving rule's
    size (N / 2500, a power of two) or half or twice as many, odd meshes and column counts among
    them."""
    kind = rng.choice(["step", "step", "step", "solve", "solve", "chamber", "request", "matvec", "matvec_c64"])
    r = rng.choice([1, 2, 2, 3])
    top = {"step": 26000, "solve": 60000, "chamber": 30000, "request": 9000, "matvec": 120000, "matvec_c64": 200000}[kind]
    target = math.exp(rng.uniform(math.log(900), math.log(top)))
    n = 2
    while _ndof(n + 1, r) <= target:
        n += 1
    overlap = rng.choice([0, 1, 1, 2]) if kind in ("step", "solve") and target < 15000 else (1 if kind in ("step", "chamber", "request") else 0)
    nsub = max(1, 2 ** max(0, math.ceil(math.log2(_ndof(n, r) / 2500.0)))) * rng.choice([1, 1, 2])
    if nsub > 4 and rng.random() < 0.3:
        nsub -= 1
    bits = 64 if kind in ("step", "solve") and r == 1 and target < 4000 and rng.random() < 0.7 else 32
    if kind == "chamber":
        k = 4 * rng.choice([1, 2, 4])
    elif bits == 64:
        k = 1
    else:
        k = rng.choice([1, 1, 2, 3, 5, 8, 12, 16, 32]) if target < 15000 or kind[:6] == "matvec" else rng.choice([1, 3, 8])
    return dict(kind=kind, n=n, r=r, nsub=nsub, overlap=overlap, k=k, bits=bits,
                restart=rng.choice([50, 50, 100, 30]), panel=rng.choice([0, 0, 24]))


# ------------------------------------------------------------------ inputs
def _ndof(n, r):
    e = 3 * n * (n + 1) ** 2 + 3 * n * n * (n + 1) + n ** 3
    t = 6 * n ** 3
    f = 1 - (n + 1) ** 3 + e + t
    return r * e + r * (r - 1) * f + r * (r - 1) * (r - 2) // 2 * t


def _mesh(n):
    """Vertex i + (n+1) (j + (n+1) k) at (i, j, k) / n; per cube the six tetrahedra along the paths
    from its lowest to its highest corner.  Vertices of each tetrahedron are ascending."""
    m = n + 1
    g = np.arange(m) / n
    kk, jj, ii = np.meshgrid(g, g, g, indexing="ij")
    xyz = np.stack([ii.ravel(), jj.ravel(), kk.ravel()], axis=1)
    ck, cj, ci = np.meshgrid(np.arange(n), np.arange(n), np.arange(n), indexing="ij")
    c = (ci + m * (cj + m * ck)).ravel()
    step = (1, m, m * m)
    paths = [np.cumsum([0] + [step[a] for a in p]) for p in itertools.permutations(range(3))]
    tets = np.stack([c[:, None] + p[None, :] for p in paths], axis=1).reshape(-1, 4)
    return xyz, tets.astype(np.int32)


def _materials(xyz, tets, rng):
    c = xyz[tets].mean(axis=1)
    eps = np.full(len(tets), EPS_GEL)
    eps[np.linalg.norm(c - 0.5, axis=1) < 0.35] = complex(40.0, -15.0)
    at = np.array([0.5 + 0.1 * rng.uniform(-1, 1), 0.5, 0.5])
    eps[np.linalg.norm(c - at, axis=1) < rng.uniform(0.06, 0.12)] = complex(rng.uniform(50, 70), -rng.uniform(15, 30))
    return eps * (1.0 + 1e-3 * rng.uniform(-1, 1, len(tets)))


def _dipoles(rng, k):
    th = 2.0 * math.pi * (np.arange(k) + rng.uniform(0.05, 0.95)) / k
    pts = np.stack([0.5 + 0.45 * np.cos(th), 0.5 + 0.45 * np.sin(th), np.full(k, 0.4871) + 0.02 * rng.uniform(0, 1, k)], axis=1)
    return pts, np.array([0.0, 0.0, 1.0])


def _inputs(case, seed):
    rng = np.random.default_rng(seed)
    xyz, tets = _mesh(case["n"])
    eps = _materials(xyz, tets, rng)
    pts, d = _dipoles(rng, case["k"])
    return xyz, tets, eps, pts, d


class State:
    """What a program keeps: the handle with its factors, and its buffers."""

    def __init__(self, case):
        self.kind, self.case, self.h = case["kind"], case, None

    def __del__(self):
        if self.h is not None:
            O.oras_destroy(self.h)
            self.h = None


def _options(case):
    return dict(restart=case["restart"], factor_bits=case["bits"], lu_panel=case["panel"])


def _ports(k):
    """k ports of the four side faces of the unit cube: k / 4 strips of width 1 per face, the TE10
    mode across them."""
    q, out = k // 4, []
    for a in range(q):
        z, dz = a / q, 1.0 / q
        for origin, u in (((0, 0, z), (1, 0, 0)), ((0, 1, z), (1, 0, 0)), ((0, 0, z), (0, 1, 0)), ((1, 0, z), (0, 1, 0))):
            out.append((origin, u, (0.0, 0.0, dz)))
    return out


def prepare(case, seed):
    s = State(case)
    xyz, tets, eps, pts, d = _inputs(case, seed)
    k, r = case["k"], case["r"]
    if s.kind == "request":
        s.args = (xyz, tets, eps, None, K0, r, case["nsub"], case["overlap"])
        s.pts, s.d = pts, d
        return s
    if s.kind == "chamber":
        # metallic bottom, ports on the four sides (their propagation constant on those faces)
        beta = math.sqrt(59.0 * K0 * K0 - math.pi ** 2)
        faces = np.stack([xyz[np.delete(tets, q, axis=1)] for q in range(4)], axis=1)   # opposite vertex q
        on = lambda ax, val: np.all(faces[:, :, :, ax] == val, axis=2)  # noqa: E731
        kind = on(2, 0.0).astype(np.uint8)
        side = on(0, 0.0) | on(0, 1.0) | on(1, 0.0) | on(1, 1.0)
        bf = np.where(side, beta, K0 * math.sqrt(EPS_GEL.real))
        s.h = O.oras_create(xyz, tets, r, case["nsub"], case["overlap"], beta_face=bf, face_kind=kind, **_options(case))
        s.ports = [O.port(o, u, v, beta) for o, u, v in _ports(k)]
    else:
        s.h = O.oras_create(xyz, tets, r, case["nsub"], case["overlap"], **_options(case))
    s.eps = torch.from_numpy(eps).cuda()
    O.oras_factor(s.h, s.eps, None, K0, mem=O.ORAS_MEM_DEVICE)
    n = O.oras_ndof(s.h)
    s.b = torch.empty(k, n, dtype=torch.complex128, device="cuda")
    s.x = torch.empty_like(s.b)
    if s.kind == "chamber":
        for j, p in enumerate(s.ports):
            s.b[j] = torch.from_numpy(O.oras_rhs_port(s.h, p)).cuda()
    elif s.kind in ("matvec", "matvec_c64"):
        g = torch.Generator(device="cuda").manual_seed(int(seed))
        v = torch.randn(k, n, 2, dtype=torch.float64, device="cuda", generator=g)
        s.b = torch.view_as_complex(v)
        if s.kind == "matvec_c64":
            s.b = s.b.to(torch.complex64)
    else:
        for j in range(k):
            O.oras_rhs_dipole(s.h, pts[j], d, mem=O.ORAS_MEM_DEVICE, out=s.b[j])
    return s


def run(s):
    k, dev = s.case["k"], O.ORAS_MEM_DEVICE
    if s.kind == "request":
        h = O.oras_setup(*s.args, **_options(s.case))
        try:
            b = np.stack([O.oras_rhs_dipole(h, p, s.d) for p in s.pts], axis=1)
            x, _, _ = O.oras_solve(h, b, TOL, k=k)
        finally:
            O.oras_destroy(h)
        return x
    if s.kind == "matvec":
        return O.oras_matvec(s.h, s.b, k=k, mem=dev, out=s.x)
    if s.kind == "matvec_c64":
        return O.oras_matvec_c64(s.h, s.b, k=k, mem=dev, out=s.x)
    if s.kind in ("step", "chamber"):
        O.oras_factor(s.h, s.eps, None, K0, mem=dev)
    x, _, _ = O.oras_solve(s.h, s.b, TOL, k=k, mem=dev, out=s.x)
    if s.kind == "chamber":
        return x, O.oras_s_matrix(s.h, s.ports, x.cpu().numpy().T)
    return x


def work(case):
    """The data in and out and A once, and one product with A a column (an iteration's least)."""
    N, k = _ndof(case["n"], case["r"]), case["k"]
    nnz = NNZ_ROW[case["r"]] * N
    io = (24 if case["kind"] == "matvec_c64" else 32) * N * k
    return {"bytes": io + 20.0 * nnz, "flops": 8.0 * nnz * k}


# ------------------------------------------------------------------ the same in plain numpy, 64 bits
E6 = ((0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3))
F4 = ((0, 1, 2), (0, 1, 3), (0, 2, 3), (1, 2, 3))


def _generators(r):
    """(kind, entity, i, j, exponents): lambda^k (lambda_i grad lambda_j - lambda_j grad lambda_i)."""
    def powers(on):
        out = []
        for p in itertools.product(range(r), repeat=len(on)):
            if sum(p) == r - 1:
                e = [0, 0, 0, 0]
                for v, q in zip(on, p):
                    e[v] = q
                out.append(tuple(e))
        return out
    gen = [("e", q, a, b, p) for q, (a, b) in enumerate(E6) for p in powers((a, b))]
    for q, (a, b, c) in enumerate(F4):
        for i, j, o in ((a, b, c), (a, c, b)):
            gen += [("f", q, i, j, p) for p in powers((a, b, c)) if p[o] >= 1]
    if r == 3:
        for i, j in ((0, 1), (0, 2), (0, 3)):
            gen.append(("v", 0, i, j, tuple(int(v not in (i, j)) for v in range(4))))
    return gen


def _numbering(tets, r, gen):
    m = int(tets.max()) + 1
    st = tets.astype(np.int64)
    ek, ei = np.unique(np.stack([st[:, a] * m + st[:, b] for a, b in E6], axis=1), return_inverse=True)
    fk, fi = np.unique(np.stack([(st[:, a] * m + st[:, b]) * m + st[:, c] for a, b, c in F4], axis=1), return_inverse=True)
    ei, fi = ei.reshape(-1, 6), fi.reshape(-1, 4)
    ne, nf = r, r * (r - 1)
    cols, seen = [], {}
    for kind, q, *_ in gen:
        i = seen.get((kind, q), 0)
        seen[(kind, q)] = i + 1
        if kind == "e":
            cols.append(ei[:, q] * ne + i)
        elif kind == "f":
            cols.append(len(ek) * ne + fi[:, q] * nf + i)
        else:
            cols.append(len(ek) * ne + len(fk) * nf + np.arange(len(st)) * 3 + i)
    outer = np.bincount(fi.ravel())[fi] == 1
    return np.stack(cols, axis=1), outer


def _grads(p):
    inv = np.linalg.inv((p[1:] - p[0]).T)
    return np.concatenate([-inv.sum(axis=0, keepdims=True), inv])


def _values(gen, lam, gl):
    """Values and curls of the generators at barycentric points lam [P, 4]: [nl, P, 3] each."""
    w, c = [], []
    for _, _, i, j, p in gen:
        p = np.array(p)
        mono = np.prod(lam ** p, axis=1)[:, None]
        grad = sum(p[v] * (lam[:, v] ** max(p[v] - 1, 0) * np.prod(np.delete(lam ** p, v, axis=1), axis=1))[:, None] * gl[v]
                   for v in range(4))
        wh = lam[:, i:i + 1] * gl[j] - lam[:, j:j + 1] * gl[i]
        w.append(mono * wh)
        c.append(np.cross(grad, wh) + 2.0 * mono * np.cross(gl[i], gl[j]))
    return np.array(w), np.array(c)


def _simplex_points(d, q=8):
    """Collapsed Gauss-Legendre points of a d-simplex: barycentrics [P, d + 1], weights of sum 1."""
    x, w = np.polynomial.legendre.leggauss(q)
    x, w = 0.5 * (x + 1.0), 0.5 * w
    lam, wt = [], []
    for ix in itertools.product(range(q), repeat=d):
        left, weight, b = 1.0, math.factorial(d), []
        for a, i in enumerate(ix):
            b.append(left * x[i])
            weight *= w[i] * (1.0 - x[i]) ** (d - 1 - a)
            left *= 1.0 - x[i]
        lam.append([left] + b)
        wt.append(weight)
    return np.array(lam), np.array(wt)


class _System:
    """A of one case, element by element (six shapes of tetrahedra)."""

    def __init__(self, case, xyz, tets, eps):
        gen = _generators(case["r"])
        self.gen, self.xyz, self.tets = gen, xyz, tets
        self.dofs, outer = _numbering(tets, case["r"], gen)
        self.N = int(self.dofs.max()) + 1
        self.parts = []                                  # (tets, matrix, scale per tet)
        lam3, w3 = _simplex_points(3)
        lam2, w2 = _simplex_points(2)
        for s in range(6):
            ts = np.arange(s, len(tets), 6)
            p = xyz[tets[s]]
            gl, vol = _grads(p), abs(np.linalg.det(p[1:] - p[0])) / 6.0
            w, c = _values(gen, lam3, gl)
            K = vol * np.einsum("apd,bpd,p->ab", c, c, w3)
            M = vol * np.einsum("apd,bpd,p->ab", w, w, w3)
            self.parts.append((ts, K, np.ones(len(ts))))
            self.parts.append((ts, M, -K0 * K0 * eps[ts]))
            for f, vs in enumerate(F4):
                tf = ts[outer[ts, f]]
                if not len(tf):
                    continue
                lam = np.zeros((len(lam2), 4))
                lam[:, vs] = lam2
                nrm = np.cross(p[vs[1]] - p[vs[0]], p[vs[2]] - p[vs[0]])
                area = 0.5 * np.linalg.norm(nrm)
                t = np.cross(_values(gen, lam, gl)[0], nrm / (2.0 * area))
                self.parts.append((tf, area * np.einsum("apd,bpd,p->ab", t, t, w2), 1j * K0 * np.sqrt(eps[tf].real)))

    def times(self, x):                                  # [k, N] -> [k, N]
        y = np.zeros(x.shape, dtype=np.complex128)
        for ts, B, sc in self.parts:
            g = self.dofs[ts]
            v = (x[:, g] @ B) * sc[None, :, None]
            for j in range(len(x)):
                y[j] += np.bincount(g.ravel(), v[j].real.ravel(), self.N) + 1j * np.bincount(g.ravel(), v[j].imag.ravel(), self.N)
        return y

    def dense(self):
        A = np.zeros((self.N, self.N), dtype=np.complex128)
        for ts, B, sc in self.parts:
            g = self.dofs[ts]
            np.add.at(A, (g[:, :, None], g[:, None, :]), sc[:, None, None] * B[None])
        return A

    def dipole(self, x0, d):
        for t in range(len(self.tets)):
            p = self.xyz[self.tets[t]]
            gl = _grads(p)
            lam = gl @ (x0 - p[0])
            lam[0] += 1.0
            if lam.min() >= -1e-12:
                b = np.zeros(self.N, dtype=np.complex128)
                b[self.dofs[t]] = _values(self.gen, lam[None, :], gl)[0][:, 0, :] @ d
                return b
        raise ValueError("the dipole lies outside the mesh")


def exact(case, seed):
    """The products with A, and the fields of the problems small enough for a dense solve."""
    kind = case["kind"]
    xyz, tets, eps, pts, d = _inputs(case, seed)
    if kind in ("matvec", "matvec_c64"):
        if _ndof(case["n"], case["r"]) * case["k"] > 4_000_000:
            return None
        S = _System(case, xyz, tets, eps)
        g = torch.Generator(device="cuda").manual_seed(int(seed))
        v = torch.view_as_complex(torch.randn(case["k"], S.N, 2, dtype=torch.float64, device="cuda", generator=g))
        if kind == "matvec_c64":
            v = v.to(torch.complex64)
        return torch.from_numpy(S.times(v.cpu().numpy().astype(np.complex128)))
    if kind == "chamber" or _ndof(case["n"], case["r"]) > 7000:
        return None
    S = _System(case, xyz, tets, eps)
    B = np.stack([S.dipole(p, d) for p in pts], axis=1)
    X = np.linalg.solve(S.dense(), B)
    if kind == "request":
        return X if case["k"] > 1 else X[:, 0]
    return torch.from_numpy(np.ascontiguousarray(X.T))
