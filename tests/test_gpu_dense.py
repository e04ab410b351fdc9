"""The dense local factors (lu_engine=ORAS_LU_CUDA_CORES): LU with tournament pivoting over whole columns, its tensor-core
and CUDA-core applies, the allocation-free apply in the fixed array, and the panel widths, against the oracle.

Bars, as for the FP32 dense factors elsewhere: 10 * 2^-11 for products with TF32 operands against the CUDA-core apply of
the same factors, and on top of that apply's own distance from the oracle; 10 * 2^-11 (20 * 2^-11 at degree 3) for FP32
factors against the oracle; 1e-9 for FP64 factors.
"""
import functools

import numpy as np
import pytest

import synth
from oracle import dd, problem

pytestmark = pytest.mark.gpu

TF32 = 10 * 2.0 ** -11


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


@functools.lru_cache(maxsize=1)
def oracle(n, r, nsub, overlap):
    return problem.from_workload(synth.small(n=n, r=r, nsub=nsub, overlap=overlap))


def dense(O, w, **kw):
    xyz, tets = w.mesh()
    eps, mu = w.materials(xyz, tets)
    return O.oras_setup(xyz, tets, eps, mu, w.k0, w.r, w.nsub, w.overlap, restart=w.restart,
                        lu_engine=O.ORAS_LU_CUDA_CORES, **kw)


# one tile a subdomain; odd and even tile counts; 40 tiles and more; one CTA a subdomain (at least one for every SM)
@pytest.mark.parametrize("k", [8, 11, 16, 32])
@pytest.mark.parametrize("n,r,nsub,delta", [(4, 2, 8, 1), (3, 3, 4, 1), (4, 1, 64, 0), (6, 2, 2, 1), (10, 2, 256, 1)])
def test_tensor_core_apply(O, n, r, nsub, delta, k):
    w = synth.small(n=n, r=r, nsub=nsub, overlap=delta)
    p = oracle(n, r, nsub, delta)
    hs = [dense(O, w, apply_engine=e) for e in (O.ORAS_APPLY_AUTO, O.ORAS_APPLY_CUDA_CORES)]
    try:
        rng = np.random.default_rng(1000 * k + n)
        V = rng.normal(size=(p.topo.ndof, k)) + 1j * rng.normal(size=(p.topo.ndof, k))
        T, C = (O.oras_precond(h, V, k=k) for h in hs)
        assert not np.array_equal(T, C)                     # two kernels
        for j in range(k):
            assert rel(T[:, j], C[:, j]) <= TF32
        for j in (0, k // 2, k - 1):
            z = p.oras.apply(V[:, j])
            assert rel(C[:, j], z) <= 2 * TF32
            assert rel(T[:, j], z) <= rel(C[:, j], z) + TF32
    finally:
        for h in hs:
            O.oras_destroy(h)


def test_tensor_core_apply_without_partition_of_unity(O):
    w = synth.small(n=4, r=2, nsub=8, overlap=1)
    p = problem.from_workload(w)
    oas = dd.ORAS(p.topo, p.xyz, p.eps_r, p.mu_r, p.k0, p.dec, weights="none")
    h = dense(O, w, weights=O.ORAS_WEIGHTS_NONE)
    try:
        rng = np.random.default_rng(77)
        V = rng.normal(size=(p.topo.ndof, 16)) + 1j * rng.normal(size=(p.topo.ndof, 16))
        Z = O.oras_precond(h, V, k=16)
        for j in (0, 7, 15):
            assert rel(Z[:, j], oas.apply(V[:, j])) <= 2 * TF32
    finally:
        O.oras_destroy(h)


@pytest.mark.parametrize("n,nsub,overlap,bits,panel", [
    (3, 1, 0, 64, 0), (3, 1, 0, 64, 2), (3, 1, 0, 32, 3), (3, 1, 0, 32, 24), (3, 1, 0, 32, 12), (3, 1, 0, 32, 20),
    (3, 1, 0, 64, 20), (4, 8, 1, 64, 0), (4, 8, 1, 32, 0), (4, 8, 1, 32, 2), (4, 8, 1, 64, 24)])
def test_interchanges_across_panels(O, n, nsub, overlap, bits, panel):
    """Degree 3, whose local matrices take their pivots from beyond the panel; panels that end on a part of a sub-panel."""
    w = synth.small(n=n, r=3, nsub=nsub, overlap=overlap)
    p = problem.from_workload(w)
    h = dense(O, w, factor_bits=bits, lu_panel=panel)
    try:
        rng = np.random.default_rng(31)
        v = rng.normal(size=p.topo.ndof) + 1j * rng.normal(size=p.topo.ndof)
        assert rel(O.oras_precond(h, v), p.oras.apply(v)) <= (1e-9 if bits == 64 else 2 * TF32)
    finally:
        O.oras_destroy(h)


@pytest.mark.parametrize("bits,weights", [(32, 0), (64, 0), (32, 1)])
@pytest.mark.parametrize("n,nsub,overlap", [(4, 8, 1), (6, 128, 0)])
def test_allocation_free_apply(O, n, nsub, overlap, bits, weights):
    """The fixed array against the regular apply, two calls in a row; more subdomains than pairs of SMs."""
    import torch
    w = synth.small(n=n, r=2, nsub=nsub, overlap=overlap)
    h = dense(O, w, factor_bits=bits, weights=weights)
    try:
        N = O.oras_ndof(h)
        rng = np.random.default_rng(bits)
        for k in (1, 2):
            V = rng.normal(size=(k, N)) + 1j * rng.normal(size=(k, N))
            ref = np.asarray(O.oras_precond(h, V.T.copy(), k=k)).reshape(N, k)
            vd = torch.from_numpy(V).cuda()
            zd = torch.full_like(vd, complex(np.nan, np.nan))
            O.oras_precond_noalloc(h, vd, zd, k)
            torch.cuda.synchronize()
            # strips may be summed in another order
            assert rel(zd.cpu().numpy().T, ref) <= (1e-12 if bits == 64 else 1e-5)
    finally:
        O.oras_destroy(h)


def test_local_vectors_in_global_memory(O):
    """One subdomain of 21,000 unknowns: a cluster of four CTAs, whose vectors are in shared memory for one right-hand side
    and in global memory for four."""
    w = synth.small(n=8, r=2, nsub=1, overlap=0)
    h = dense(O, w)
    try:
        N = O.oras_ndof(h)
        assert O.oras_subdomain_size(h, 0)[2] > 20000
        rng = np.random.default_rng(22)
        V = rng.normal(size=(N, 6)) + 1j * rng.normal(size=(N, 6))
        Z = O.oras_precond(h, V, k=6)
        for j in range(6):
            assert rel(Z[:, j], O.oras_precond(h, V[:, j].copy())) <= 1e-5
            assert np.linalg.norm(V[:, j] - O.oras_matvec(h, Z[:, j].copy())) <= 1e-2 * np.linalg.norm(V[:, j])
    finally:
        O.oras_destroy(h)


def test_autotuned_panel_width(O):
    w = synth.small(n=5, r=2, nsub=4, overlap=1)
    p = problem.from_workload(w)
    h = dense(O, w)
    try:
        panel, times = O.oras_autotune(h)
        assert panel in O.AUTOTUNE_WIDTHS and len(times) == len(O.AUTOTUNE_WIDTHS) + 3
        rng = np.random.default_rng(8)
        v = rng.normal(size=p.topo.ndof) + 1j * rng.normal(size=p.topo.ndof)
        assert rel(O.oras_precond(h, v), p.oras.apply(v)) <= TF32
    finally:
        O.oras_destroy(h)
