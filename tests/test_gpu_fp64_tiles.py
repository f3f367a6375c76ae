"""FP64 tile kernels at the edges of their tiles: the object operations (general strides, contraction split over
clusters, matrix-vector forms) and the FP64 J/K build on ragged sizes, against numpy.

Tolerance: a sum of k products in any order differs from the exact one by at most k eps sum|a b| (Higham,
Accuracy and Stability of Numerical Algorithms, ch. 3); two such sums by twice that."""
import numpy as np
import pytest

from paper_1707_03771_gb300 import clusters

pytestmark = pytest.mark.gpu
EPS = np.finfo(float).eps


@pytest.fixture(scope="module")
def lib():
    from paper_1707_03771_gb300 import binding, build
    build.build()
    return binding


@pytest.fixture(scope="module")
def handle(lib):
    with lib.Handle(clusters.water_cluster(1, 3)) as h:
        h.build_B()
        yield h


def _close(got, ref, absref, k):
    assert got.shape == ref.shape
    assert np.all(np.abs(got - ref) <= 2 * (k + 2) * EPS * absref + 1e-300), np.abs(got - ref).max()


@pytest.mark.parametrize("shape", [(1, 1, 1, 1), (2, 3, 1, 5), (3, 17, 16, 9), (5, 15, 65, 40), (70, 33, 41, 20),
                                   (9, 64, 129, 41), (300, 7, 31, 10)])
def test_object_operations_on_ragged_shapes(lib, handle, shape):
    naux, nr, ns, nt = shape
    rng = np.random.default_rng(naux + nr)
    I = rng.standard_normal((naux, nr, ns))
    M1, M2, Ma = rng.standard_normal((nr, nt)), rng.standard_normal((ns, nt)), rng.standard_normal((nt, naux))
    D, g = rng.standard_normal((nr, ns)), rng.standard_normal(naux)
    T = lib.DFTensor.create(handle, I)
    e = np.einsum
    for which, M, spec, k in (("first", M1, "grs,rt->gts", nr), ("second", M2, "grs,st->grt", ns), ("aux", Ma, "tg,grs->trs", naux)):
        out = T.transform(which, M)
        ops = (M, I) if which == "aux" else (I, M)
        _close(out.get(), e(spec, *ops), e(spec, *map(np.abs, ops)), k)
        out.close()
    for which, spec, k in (("first", "grs,grt->st", naux * nr), ("pairs", "grs,drs->gd", nr * ns)):
        _close(T.contract(T, which), e(spec, I, I), e(spec, np.abs(I), np.abs(I)), k)
    if nr * ns <= 700:
        _close(T.contract(T, "aux"), I.reshape(naux, -1).T @ I.reshape(naux, -1),
               np.abs(I).reshape(naux, -1).T @ np.abs(I).reshape(naux, -1), naux)
    _close(T.density_fit(D), e("grs,rs->g", I, D), e("grs,rs->g", np.abs(I), np.abs(D)), nr * ns)
    _close(T.density_back(g), e("g,grs->rs", g, I), e("g,grs->rs", np.abs(g), np.abs(I)), naux)
    T.close()


@pytest.mark.parametrize("nocc", [1, 5, 7, 10, 13, 33, 41, 50])
def test_fp64_exchange_for_any_number_of_orbitals(lib, handle, nocc):
    n, naux = handle.n, handle.naux
    rng = np.random.default_rng(nocc)
    C = rng.standard_normal((n, nocc))
    B = handle.rows(1, 0, naux)
    J, K = handle.jk(C @ C.T, C)
    Y, Ya = B @ C, np.abs(B) @ np.abs(C)
    _close(K, np.einsum("gmi,gni->mn", Y, Y), np.einsum("gmi,gni->mn", Ya, Ya), naux * nocc + 2 * n)
    assert np.array_equal(K, K.T)
