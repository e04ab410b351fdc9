"""The sparse local factors (block L D L^T over an elimination tree, pivots inside a tree node) against
the dense LU with pivoting over whole columns (lu_engine CUDA_CORES) of the same matrices, and against
the oracle's ORAS (Sec. 4), over the forms oras_create accepts.

FP32 bars: the factors round at 2^-24, amplified by the condition number of the local matrices (1e3 to
4e3 at degrees 1 and 2 in the lossy medium, up to 3e4 at degree 3 and 7e4 without losses): 2^-24 cond,
3e-4 at degrees 1 and 2, 5e-3 else.  FP64: 1e-9, as for every FP64 apply.
"""
import numpy as np
import pytest

import synth
from oracle import dd, problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def O():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1605_04521_gb300 import build
    build.build()
    from paper_1605_04521_gb300 import oras
    return oras


def rel(a, b):
    return np.linalg.norm(np.ravel(a) - np.ravel(b)) / max(np.linalg.norm(np.ravel(b)), 1e-300)


def shuffled(xyz, tets, seed):
    """The same mesh with its vertices renumbered, its tetrahedra reordered and their vertices permuted."""
    rng = np.random.default_rng(seed)
    p = rng.permutation(len(xyz))
    t = p[tets][rng.permutation(len(tets))]
    x = np.empty_like(xyz)
    x[p] = xyz
    return x, np.ascontiguousarray(rng.permuted(t, axis=1)).astype(np.int32)


CASES = {
    # one node a subdomain (19-dof tetrahedra groups); odd and single subdomains; chains of pivot blocks
    "one_node": dict(n=3, r=1, nsub=54, ov=0),
    "one_subdomain": dict(n=4, r=2, nsub=1, ov=0),
    "odd_subdomains": dict(n=4, r=1, nsub=7, ov=2),
    "degree3": dict(n=3, r=3, nsub=5, ov=1),
    # unstructured numbering, a random partition (disconnected subdomains), face overlap
    "shuffled": dict(n=4, r=2, nsub=6, ov=1, shuffle=3),
    "random_partition": dict(n=3, r=2, nsub=6, ov=0, shuffle=4, random_part=True),
    "face_overlap": dict(n=4, r=2, nsub=5, ov=1, opts=dict(overlap_kind=1)),
    # R_s A R_s^T couples unknowns through tetrahedra outside the subdomain
    "dirichlet": dict(n=4, r=2, nsub=6, ov=1, opts=dict(transmission=1)),
    "dirichlet_random_partition": dict(n=3, r=1, nsub=5, ov=0, shuffle=5, random_part=True, opts=dict(transmission=1)),
    "oas": dict(n=4, r=2, nsub=6, ov=1, opts=dict(weights=1)),
    "metallic": dict(n=4, r=2, nsub=6, ov=1, metal=True),
    "lossless": dict(n=4, r=2, nsub=4, ov=1, eps=4.0, k0=2.5),
}


@pytest.mark.parametrize("bits", [32, 64])
@pytest.mark.parametrize("name", sorted(CASES))
def test_sparse_factors_match_dense_lu_and_oracle(O, name, bits):
    c = CASES[name]
    xyz, tets = synth.kuhn_cube(c["n"])
    if "shuffle" in c:
        xyz, tets = shuffled(xyz, tets, c["shuffle"])
    nt, r, nsub, ov = len(tets), c["r"], c["nsub"], c["ov"]
    eps, mu = synth.head_materials(xyz, tets) if "eps" not in c else (np.full(nt, c["eps"] + 0j), np.ones(nt, complex))
    k0, opts = c.get("k0", synth.K0), c.get("opts", {})
    part = None
    if c.get("random_part"):
        part = np.random.default_rng(9).permutation(np.arange(nt) % nsub).astype(np.int32)
    kind = None
    if c.get("metal"):
        faces = np.stack([xyz[np.delete(tets, q, axis=1)] for q in range(4)], axis=1)
        kind = np.all(faces[:, :, :, 2] == 0.0, axis=2).astype(np.uint8)
    hs = [O.oras_setup(xyz, tets, eps, mu, k0, r, nsub, ov, part=part, face_kind=kind, factor_bits=bits, lu_engine=e, **opts)
          for e in (O.ORAS_LU_AUTO, O.ORAS_LU_CUDA_CORES)]
    try:
        n = O.oras_ndof(hs[0])
        rng = np.random.default_rng(7)
        bar = 1e-9 if bits == 64 else (5e-3 if r == 3 or name == "lossless" else 3e-4)
        prob = problem.build(xyz, tets, eps, mu, k0, r, [], nsub=nsub, delta=ov, part=part, face_kind=kind,
                             with_oras=not opts)
        orac = prob.oras
        if "overlap_kind" not in opts and opts:
            dec = dd.decompose(prob.topo, xyz, nsub, ov, part)
            orac = dd.ORAS(prob.topo, xyz, eps, mu, k0, dec, weights="none" if "weights" in opts else "pou",
                           transmission="dirichlet" if "transmission" in opts else "impedance", A_global=prob.A.tocsr())
        for k in (1, 2, 3, 5, 8, 11):  # every group size, full and partly used
            V = rng.normal(size=(n, k)) + 1j * rng.normal(size=(n, k))
            Z, D = (np.asarray(O.oras_precond(h, V, k=k)).reshape(n, k) for h in hs)
            for j in range(k):
                # many columns on the dense FP32 factors go through TF32 products: against the oracle only
                if bits == 64 or k < 8:
                    assert rel(Z[:, j], D[:, j]) <= bar
                if orac is not None:
                    assert rel(Z[:, j], orac.apply(V[:, j])) <= bar
    finally:
        for h in hs:
            O.oras_destroy(h)


@pytest.mark.parametrize("nsub", [1, 2])
def test_half_dead_medium_stays_singular(O, nsub):
    """eps_r = 0 and 1/mu_r = 0 in half of the tetrahedra make local matrices with exactly zero rows: refused
    with one subdomain over both halves and with one each, as by the dense LU."""
    xyz, tets = synth.kuhn_cube(3)
    nt = len(tets)
    dead = xyz[tets].mean(axis=1)[:, 0] < 0.5
    eps = np.where(dead, 0.0, 44.0 - 20.0j)
    mu = np.where(dead, 1e300, 1.0).astype(complex)
    part = (dead.astype(np.int32) if nsub == 2 else np.zeros(nt, dtype=np.int32))
    for engine in (O.ORAS_LU_AUTO, O.ORAS_LU_CUDA_CORES):
        with pytest.raises(O.OrasError) as e:
            O.oras_setup(xyz, tets, eps, mu, synth.K0, 2, nsub, 0, part=part, lu_engine=engine)
        assert e.value.code == O.ORAS_ERR_SINGULAR_LOCAL


@pytest.mark.parametrize("case", ["odd_subdomains", "degree3_chains", "one_subdomain"])
def test_columns_together_equal_columns_alone(O, case):
    """One column at a time against 8, 16 and 32 a pass, full and partly used: tiles of 16 and 64 own unknowns, sums
    shorter than a stage and longer than all stages.  Bar: both sum the same FP32 products in another order, 2^-24 cond
    (as above, at degree 3 5e-3), in practice far below."""
    c = dict(odd_subdomains=dict(n=5, r=2, nsub=7, ov=1), degree3_chains=dict(n=4, r=3, nsub=3, ov=0),
             one_subdomain=dict(n=6, r=2, nsub=1, ov=0))[case]
    xyz, tets = synth.kuhn_cube(c["n"])
    eps, mu = synth.head_materials(xyz, tets)
    h = O.oras_setup(xyz, tets, eps, mu, synth.K0, c["r"], c["nsub"], c["ov"])
    try:
        n = O.oras_ndof(h)
        rng = np.random.default_rng(11)
        V = rng.normal(size=(n, 37)) + 1j * rng.normal(size=(n, 37))
        alone = np.stack([O.oras_precond(h, V[:, j]) for j in range(37)], axis=1)
        bar = 5e-3 if c["r"] == 3 else 3e-4
        for k in (5, 8, 9, 16, 17, 32, 37):
            Z = np.asarray(O.oras_precond(h, V[:, :k], k=k))
            for j in range(k):
                assert rel(Z[:, j], alone[:, j]) <= bar
    finally:
        O.oras_destroy(h)


@pytest.mark.parametrize("bits,weights", [(32, 0), (64, 0), (32, 1)])
def test_captured_noalloc_apply_outlives_larger_calls(O, bits, weights):
    """The allocation-free apply in a CUDA graph, replayed after calls with more columns have made the handle's other
    workspace grow and after new materials: the factors and vectors it uses are still where they were captured."""
    import torch
    w = synth.small(n=4, r=2, nsub=8, overlap=1)
    xyz, tets = w.mesh()
    eps, mu = w.materials(xyz, tets)
    h = O.oras_setup(xyz, tets, eps, mu, w.k0, w.r, w.nsub, w.overlap, factor_bits=bits, weights=weights)
    try:
        n = O.oras_ndof(h)
        rng = np.random.default_rng(17)
        V = rng.normal(size=(2, n)) + 1j * rng.normal(size=(2, n))
        vd = torch.from_numpy(V).cuda()
        zd = torch.zeros_like(vd)
        stream = torch.cuda.Stream()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        O.oras_set_stream(h, stream.cuda_stream)
        O.oras_precond_noalloc(h, vd, zd, 2)               # the first call on a device comes before a capture
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=stream):
            O.oras_precond_noalloc(h, vd, zd, 2)
        B = rng.normal(size=(n, 40)) + 1j * rng.normal(size=(n, 40))
        for factor in (1.0, 1.3):
            O.oras_factor(h, eps * factor, mu, w.k0)
            O.oras_precond(h, B, k=40)                     # the shared workspace grows
            ref = np.stack([O.oras_precond(h, V[j]) for j in range(2)])
            zd.fill_(complex(np.nan, np.nan))
            torch.cuda.synchronize()
            with torch.cuda.stream(stream):
                graph.replay()
            torch.cuda.synchronize()
            got = zd.cpu().numpy()
            # one column at a time on both sides: the same kernels in the same order; OAS adds with atomics
            assert rel(got, ref) <= (1e-12 if bits == 64 else (1e-6 if weights else 0.0))
    finally:
        O.oras_destroy(h)


# Lossless unit cubes at the frequency at which the interior of a tree node, its border held at zero, resonates: the lowest
# eigenvalue of (K, M) on the node's unknowns, for the trees of FP32 (a node of 82 unknowns) and FP64 (one of 42).
RESONANT = {32: 6.696048910007606, 64: 9.811005223139103}


@pytest.mark.parametrize("off", [0.0, 1e-9, 1e-7, 1e-5])
@pytest.mark.parametrize("bits", [32, 64])
def test_resonating_tree_node(O, bits, off):
    """A pivot block that is singular to rounding although A_s is not: the trees are planned anew (the factors take another
    size then), the apply stays as exact as elsewhere without losses, and one subdomain still solves at once.  New
    materials and back on the same handle."""
    xyz, tets = synth.kuhn_cube(6)
    nt, k0 = len(tets), RESONANT[bits] * (1.0 + off)
    eps, mu = np.full(nt, 4.0 + 0j), np.ones(nt, complex)
    p = problem.build(xyz, tets, eps, mu, k0, 2, [("dipole", np.array([0.31, 0.45, 0.52]), np.array([0.0, 0.0, 1.0]))],
                      nsub=1, delta=0)
    rng = np.random.default_rng(3)
    v = rng.normal(size=p.topo.ndof) + 1j * rng.normal(size=p.topo.ndof)
    z = p.oras.apply(v)
    h = O.oras_create(xyz, tets, 2, 1, 0, factor_bits=bits)
    try:
        O.oras_factor(h, eps * 1.1, None, k0)
        regular = O.oras_arena_bytes(h)
        for _ in range(2):
            O.oras_factor(h, eps, None, k0)
            if off == 0.0:
                assert O.oras_arena_bytes(h) != regular
            assert rel(O.oras_precond(h, v), z) <= (1e-9 if bits == 64 else 5e-3)
            x, info, rc = O.oras_solve(h, p.B[:, 0], 1e-10)
            assert rc == O.ORAS_OK and info[0]["iterations"] <= (2 if bits == 64 else 5)
            O.oras_factor(h, eps * 1.1, None, k0)
    finally:
        O.oras_destroy(h)


@pytest.mark.parametrize("bits", [32, 64])
@pytest.mark.parametrize("nsub", [1, 3])
def test_dead_cube_in_a_live_medium_stays_singular(O, bits, nsub):
    """Six tetrahedra without any term (eps_r = 0, 1/mu_r = 0): the unknowns inside them have zero rows, in pivot blocks
    whose other unknowns are alive.  Refused, as by the dense LU."""
    n = 4
    xyz, tets = synth.kuhn_cube(n)
    dead = np.all(np.floor(xyz[tets].mean(axis=1) * n) == 1, axis=1)
    assert dead.sum() == 6
    eps = np.where(dead, 0.0, 44.0 - 20.0j)
    mu = np.where(dead, 1e300, 1.0).astype(complex)
    for engine in (O.ORAS_LU_AUTO, O.ORAS_LU_CUDA_CORES):
        with pytest.raises(O.OrasError) as e:
            O.oras_setup(xyz, tets, eps, mu, synth.K0, 2, nsub, 1, factor_bits=bits, lu_engine=engine)
        assert e.value.code == O.ORAS_ERR_SINGULAR_LOCAL and "zero pivot" in str(e.value)


@pytest.mark.parametrize("bits,power", [(32, -80), (32, -60), (32, 64), (32, 80), (64, -300), (64, -140), (64, 140), (64, 300)])
def test_entries_of_any_scale(O, bits, power):
    """A and A_s times a power of two (the mesh's unit, 1 / mu_r), far from 1 but inside the factors' precision: the apply
    is the same times its inverse.  Squares of such entries over- or underflow."""
    s = 2.0 ** power
    xyz, tets = synth.kuhn_cube(4)
    eps, mu = synth.head_materials(xyz, tets)
    beta = np.full((len(tets), 4), 9.0)
    rng = np.random.default_rng(5)
    zs = []
    for f in (1.0, s):
        # one subdomain: no interface whose coefficient comes from the materials
        h = O.oras_setup(xyz, tets, eps * f, mu / f, synth.K0, 2, 1, 0, beta_face=beta * f, factor_bits=bits)
        try:
            n = O.oras_ndof(h)
            if not zs:
                v = rng.normal(size=n) + 1j * rng.normal(size=n)
            zs.append(O.oras_precond(h, v) * f)
            x, info, rc = O.oras_solve(h, v, 1e-8)
            assert rc == O.ORAS_OK and info[0]["iterations"] <= 3
        finally:
            O.oras_destroy(h)
    assert np.all(np.isfinite(zs[1]))
    assert rel(zs[1], zs[0]) <= (1e-12 if bits == 64 else 1e-6)


@pytest.mark.parametrize("n,r,nsub", [(4, 2, 4), (5, 1, 3), (3, 3, 2)])
@pytest.mark.parametrize("k0", [0.3, 0.1, 0.02])
def test_low_frequency_fp64(O, n, r, nsub, k0):
    """At low frequencies the gradients inside a tree node are all but in its pivot block's null space; L is not large
    there.  The apply with FP64 sparse factors stays within ten times the distance of the dense LU of the same matrices
    from the oracle, or 1e-12."""
    xyz, tets = synth.kuhn_cube(n)
    eps, mu = synth.head_materials(xyz, tets)
    p = problem.build(xyz, tets, eps, mu, k0, r, [], nsub=nsub, delta=1)
    rng = np.random.default_rng(6)
    v = rng.normal(size=p.topo.ndof) + 1j * rng.normal(size=p.topo.ndof)
    z = p.oras.apply(v)
    err = []
    for engine in (O.ORAS_LU_AUTO, O.ORAS_LU_CUDA_CORES):
        h = O.oras_setup(xyz, tets, eps, mu, k0, r, nsub, 1, factor_bits=64, lu_engine=engine)
        try:
            err.append(rel(O.oras_precond(h, v), z))
        finally:
            O.oras_destroy(h)
    assert err[0] <= max(10.0 * err[1], 1e-12), err


def test_new_trees_under_captured_steps(O):
    """Arnoldi steps captured with one plan, then materials at a resonance, which change the plan: the steps are captured
    anew, and the fields are those of a handle without graphs, bit for bit."""
    import torch
    xyz, tets = synth.kuhn_cube(6)
    nt, k0 = len(tets), RESONANT[32]
    eps = np.full(nt, 4.0 + 0j)
    stream = torch.cuda.Stream()
    fields, arenas = [], []
    for graphs in (0, 1):
        h = O.oras_create(xyz, tets, 2, 1, 0, restart=4, graphs=graphs)
        try:
            O.oras_set_stream(h, stream.cuda_stream)
            for f in (1.1, 1.0, 1.0, 1.1):
                O.oras_factor(h, eps * f, None, k0)
                b = O.oras_rhs_dipole(h, [0.31, 0.45, 0.52], [0.0, 0.0, 1.0])
                for _ in range(3):                       # direct, captured, replayed
                    x, _, rc = O.oras_solve(h, b, 1e-11)
                    assert rc == O.ORAS_OK
                    fields.append(x)
                arenas.append(O.oras_arena_bytes(h))
        finally:
            O.oras_destroy(h)
    assert arenas[0] != arenas[1] == arenas[2] == arenas[3] and arenas[:4] == arenas[4:]
    assert all(np.array_equal(a, b) for a, b in zip(fields[:12], fields[12:]))
