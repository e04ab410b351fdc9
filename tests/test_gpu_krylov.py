"""Krylov kernels over the column counts where their lane and block layouts change: 1, 2, 3-4 and 5-8 right-hand
sides a group, several groups, counts that do not divide a warp, more than 32.

Bars: products with A 1e-13 relative per column, as in test_gpu_parity.py; solves 1e-8 in the true residual
against the oracle's A.
"""
import numpy as np
import pytest

import synth
from oracle import problem

pytestmark = pytest.mark.gpu

COLUMNS = [1, 2, 3, 4, 5, 7, 8, 9, 12, 17, 31, 32, 33, 64]


@pytest.fixture(scope="module")
def setup():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1605_04521_gb300 import build
    build.build()
    from paper_1605_04521_gb300 import oras as O
    w = synth.small(n=5, r=2, nsub=8, overlap=0, restart=30)
    p = problem.from_workload(w, with_oras=False)
    xyz, tets = w.mesh()
    eps, mu = w.materials(xyz, tets)
    h = O.oras_setup(xyz, tets, eps, mu, w.k0, w.r, w.nsub, w.overlap, restart=w.restart)
    yield O, h, p
    O.oras_destroy(h)


def rel(a, b):
    return np.linalg.norm(np.ravel(a) - np.ravel(b)) / max(np.linalg.norm(np.ravel(b)), 1e-300)


@pytest.mark.parametrize("k", COLUMNS)
def test_products_with_a(setup, k):
    O, h, p = setup
    rng = np.random.default_rng(k)
    X = rng.normal(size=(p.A.shape[0], k)) + 1j * rng.normal(size=(p.A.shape[0], k))
    Y = np.asarray(O.oras_matvec(h, X, k=k)).reshape(-1, k)
    Z = X.astype(np.complex64)
    Y32 = np.asarray(O.oras_matvec_c64(h, Z, k=k)).reshape(-1, k)
    R, R32 = p.A @ X, p.A @ Z.astype(np.complex128)
    for j in range(k):
        assert rel(Y[:, j], R[:, j]) <= 1e-13
        assert rel(Y32[:, j], R32[:, j]) <= 1e-13


@pytest.mark.parametrize("k", COLUMNS)
def test_blocked_orthogonalisation_in_the_solve(setup, k):
    """Random right-hand sides, one of them zero; without overlap the solve takes several blocks of 8 basis
    vectors and restarts."""
    O, h, p = setup
    rng = np.random.default_rng(100 + k)
    B = rng.normal(size=(p.A.shape[0], k)) + 1j * rng.normal(size=(p.A.shape[0], k))
    if k > 2:
        B[:, k // 2] = 0.0
    X, info, rc = O.oras_solve(h, B, 1e-8, k=k)
    X = np.asarray(X).reshape(-1, k)
    assert rc == O.ORAS_OK
    for j in range(k):
        if not B[:, j].any():
            assert not X[:, j].any()
            continue
        assert np.linalg.norm(B[:, j] - p.A @ X[:, j]) <= 1e-8 * np.linalg.norm(B[:, j])
    assert max(i["iterations"] for i in info) > 16


@pytest.mark.parametrize("k", [1, 3])
@pytest.mark.parametrize("place", ["plain", "onto_input", "half_entry"])
def test_device_vectors_wherever_they_are(setup, k, place):
    """Products of vectors given as device memory, which are read and written where they are when a kernel can and
    through a copy otherwise: the result on top of the input, both half an entry off their alignment."""
    import ctypes
    import torch
    O, h, p = setup
    n = p.A.shape[0]
    rng = np.random.default_rng(300 + k)
    X = rng.normal(size=(k, n)) + 1j * rng.normal(size=(k, n))
    for wide in (True, False):
        Z = X if wide else X.astype(np.complex64)
        R = (p.A @ Z.T.astype(np.complex128)).T
        real = torch.from_numpy(np.ascontiguousarray(Z).view(Z.real.dtype).ravel().copy())
        off = 1 if place == "half_entry" else 0
        size = 2 * k * n * (2 if not wide else 1) + off        # room for the complex128 result on top of it
        src = torch.zeros(size, dtype=real.dtype, device="cuda")
        src[off:off + len(real)] = real
        dst = torch.zeros(2 * k * n + off, dtype=torch.float64, device=src.device)
        if place == "onto_input":
            dst = src.view(torch.float64)
        at = lambda t: ctypes.c_void_p(t.data_ptr() + off * t.element_size())  # noqa: E731
        torch.cuda.synchronize()
        fn = O.lib.oras_matvec if wide else O.lib.oras_matvec_c64
        assert fn(h, at(src), at(dst), k, O.ORAS_MEM_DEVICE) == O.ORAS_OK
        torch.cuda.synchronize()
        Y = dst[off:off + 2 * k * n].cpu().numpy().view(np.complex128).reshape(k, n)
        assert rel(Y, R) <= 1e-13


@pytest.fixture(scope="module")
def larger():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1605_04521_gb300 import build
    build.build()
    from paper_1605_04521_gb300 import oras as O
    w = synth.small(n=10, r=2, nsub=16, overlap=0, restart=30)
    xyz, tets = w.mesh()
    eps, mu = w.materials(xyz, tets)
    h = O.oras_setup(xyz, tets, eps, mu, w.k0, w.r, w.nsub, w.overlap, restart=w.restart)
    yield O, h
    O.oras_destroy(h)


@pytest.mark.parametrize("k", [1, 2, 3, 5, 7, 8])
def test_orthogonalisation_in_one_launch(larger, k):
    """Up to 8 columns an Arnoldi step ends in one cooperative launch, 9 and more take several: the same columns
    through both, over several rounds of an SM's share (k entries of 1/152 of the vector, 512 at a time)."""
    O, h = larger
    n = O.oras_ndof(h)
    rng = np.random.default_rng(200 + k)
    B = rng.normal(size=(n, 9)) + 1j * rng.normal(size=(n, 9))
    Y, _, rc9 = O.oras_solve(h, B, 1e-8, k=9)
    X, info, rc = O.oras_solve(h, B[:, :k], 1e-8, k=k)
    X = np.asarray(X).reshape(-1, k)
    assert rc == rc9 == O.ORAS_OK
    assert max(i["iterations"] for i in info) > 16
    R = B[:, :k] - np.asarray(O.oras_matvec(h, X, k=k)).reshape(-1, k)
    for j in range(k):
        assert np.linalg.norm(R[:, j]) <= 1e-8 * np.linalg.norm(B[:, j])
    R9 = B[:, :k] - np.asarray(O.oras_matvec(h, np.asarray(Y)[:, :k].copy(), k=k)).reshape(-1, k)
    for j in range(k):
        assert np.linalg.norm(R9[:, j]) <= 1e-8 * np.linalg.norm(B[:, j])


def test_orthogonalisation_past_one_launch():
    """Eight columns of a vector that does not fit the SMs' shared memory (more than 18 rounds of 512 entries an SM): the
    step ends in several launches, as with more columns."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1605_04521_gb300 import build
    build.build()
    from paper_1605_04521_gb300 import oras as O
    w = synth.small(n=17, r=2, nsub=128, overlap=0, restart=20)
    xyz, tets = w.mesh()
    eps, mu = w.materials(xyz, tets)
    h = O.oras_setup(xyz, tets, eps, mu, w.k0, w.r, w.nsub, w.overlap, restart=w.restart, max_iter=18,
                     factor_bits=64)
    try:
        n = O.oras_ndof(h)
        rng = np.random.default_rng(9)
        B = rng.normal(size=(n, 8)) + 1j * rng.normal(size=(n, 8))
        launches = {}
        X = {}
        for k in (8, 1):
            O.oras_reset_timings(h)
            O.oras_set_timing(h, 1)
            X[k], info, _ = O.oras_solve(h, B[:, :k], 1e-12, k=k)
            launches[k] = O.oras_timings(h)["orth"][1]
            assert max(i["iterations"] for i in info) == 18
        assert 8 * n > 152 * 18 * 512 >= n
        assert launches[1] == 18 and launches[8] > 3 * 18
        # the same 18 steps with FP64 factors: both iterates minimise the residual over the same space, to rounding
        assert rel(np.asarray(X[8])[:, 0], np.asarray(X[1]).reshape(-1)) <= 1e-8
    finally:
        O.oras_destroy(h)


def test_grid_barrier_gives_up(setup):
    """The wait self-test includes the one-launch step's barrier, on an arrival that never comes: four waits of the limit,
    then the kernel returns and the handle works on."""
    import time
    O, _, p = setup
    w = synth.small(n=3, r=2, nsub=4, overlap=1)
    xyz, tets = w.mesh()
    eps, mu = w.materials(xyz, tets)
    h = O.oras_setup(xyz, tets, eps, mu, w.k0, w.r, w.nsub, w.overlap, wait_ms=200)
    try:
        t0 = time.perf_counter()
        rc, detail = O.oras_wait_selftest(h)
        assert time.perf_counter() - t0 >= 0.78
        assert rc == O.ORAS_ERR_DEVICE_TIMEOUT and detail == 7
        b = O.oras_rhs_dipole(h, synth.dipole_ring(1)[0], [0, 0, 1.0])
        _, info, rc = O.oras_solve(h, b, 1e-8)
        assert rc == O.ORAS_OK
    finally:
        O.oras_destroy(h)
