"""The Jacobi eigensolver by itself (dfhf::jacobi_eig on device pointers) on matrices that an SCF's Fock matrices are
not like, what a run does whose guess density is zero, and the status of a run whose grid barrier expires.

Bound. A step applies one rotation from either side to every row and column; its rounding is at most 4 eps of a pair's
norm, so a sweep of n - 1 steps adds at most 8 (n - 1) eps |A|_F to the matrix and 4 (n - 1) eps to the vectors, and at
most 12 sweeps are taken here. The elements left are below 4e-15 of the largest diagonal one, in sum below n times that."""
import ctypes
import os

import numpy as np
import pytest

from paper_1707_03771_gb300 import clusters

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


@pytest.fixture(scope="module")
def lib():
    from paper_1707_03771_gb300 import binding, build
    build.build()
    return binding


@pytest.fixture(scope="module")
def solve(lib):
    torch = pytest.importorskip("torch")
    fn = lib.load()._ZN4dfhf10jacobi_eigEP11CUstream_stiPKdPdS4_S4_Pi
    fn.restype = None
    fn.argtypes = [ctypes.c_void_p, ctypes.c_int] + [ctypes.c_void_p] * 5

    def run(A):
        n = len(A)
        a = torch.from_numpy(np.ascontiguousarray(A)).cuda()
        w = torch.empty(n, dtype=torch.float64, device="cuda")
        work = torch.empty(3 * n * n + 1, dtype=torch.float64, device="cuda")
        info = torch.full((1,), 99, dtype=torch.int32, device="cuda")
        fn(torch.cuda.current_stream().cuda_stream, n, a.data_ptr(), w.data_ptr(), a.data_ptr(), work.data_ptr(),
           info.data_ptr())
        torch.cuda.synchronize()
        return w.cpu().numpy(), a.cpu().numpy(), int(info.item())
    return run


def _matrix(kind, n):
    rng = np.random.default_rng(n)
    if kind == "zero":
        return np.zeros((n, n))
    if kind == "diagonal":
        return np.diag(rng.normal(size=n))
    if kind == "rank one":
        v = rng.normal(size=n)
        return np.outer(v, v)
    if kind == "no diagonal":
        A = rng.normal(size=(n, n))
        A = A + A.T
        np.fill_diagonal(A, 0.0)
        return A
    if kind == "degenerate":
        Q = np.linalg.qr(rng.normal(size=(n, n)))[0]
        A = (Q * np.where(np.arange(n) % 3 == 0, -20.0, 1.0)) @ Q.T
        return 0.5 * (A + A.T)
    A = rng.normal(size=(n, n)) * {"random": 1.0, "tiny": 1e-43, "tinier": 1e-250, "huge": 1e200}[kind]
    return A + A.T


@pytest.mark.parametrize("n", [1, 2, 3, 50, 199, 200])
@pytest.mark.parametrize("kind", ["zero", "diagonal", "rank one", "no diagonal", "degenerate", "random", "tiny", "tinier",
                                  "huge"])
def test_eigenpairs(solve, kind, n):
    A = _matrix(kind, n)
    w, V, info = solve(A)
    assert info == 0
    unit = max(np.abs(A).max(), np.finfo(float).tiny)          # the norms below neither over- nor underflow
    B, w = A / unit, w / unit
    assert np.all(np.diff(w) >= 0)
    steps = 12 * (n - 1)
    assert np.abs(V @ V.T - np.eye(n)).max() <= 2 * (4 * steps + n) * EPS
    off = 4e-15 * n * np.abs(w).max()
    assert np.abs(B @ V.T - V.T * w).max() <= (8 * steps + 2 * n) * EPS * np.linalg.norm(B) + off


def test_zero_guess_density(lib):
    with lib.Handle(clusters.workload("water2")) as h:
        ref = h.scf(guess="sad")
        r = h.scf(guess=np.zeros((h.n, h.n)))
    assert r["converged"] and abs(r["energy"] - ref["energy"]) < 1e-8


def test_expired_barrier_is_a_timeout(lib):
    net = lib.Mlp(5, 17, 1, 19, seed=1)
    X, Y = np.ones((3, 5), np.float32), np.ones((3, 19), np.float32)
    with lib.Handle(clusters.workload("water2")) as h:
        ref, pred = h.scf(), net.predict(X)
        os.environ["DFHF_GRID_WAIT_CYCLES"] = "1"
        try:
            with pytest.raises(lib.DFError) as e:
                h.scf()
            with pytest.raises(lib.DFError) as e2:
                net.predict(X)
            with pytest.raises(lib.DFError) as e3:
                net.gradients(X, Y)
        finally:
            del os.environ["DFHF_GRID_WAIT_CYCLES"]
        assert e.value.code == lib.DF_E_TIMEOUT and "Jacobi" in str(e.value)
        assert e2.value.code == lib.DF_E_TIMEOUT and e3.value.code == lib.DF_E_TIMEOUT
        again = h.scf()
        assert again["energy"] == ref["energy"] and np.array_equal(net.predict(X), pred)
    net.close()
