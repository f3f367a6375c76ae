"""The eigensolver of small FP64 runs (even and odd orders, up to and beyond its largest): the orbitals of a
converged SCF solve F C = S C eps and are orthonormal in S.

Tolerance: an eigensolver's residual is a small multiple of n eps |F'| in the orthogonal basis; going back through
X multiplies by |X| (smallest eigenvalue of S in these bases about 1e-3), and F is one iteration newer than the
orbitals, which the convergence thresholds bound by 1e-8."""
import numpy as np
import pytest

from paper_1707_03771_gb300 import clusters

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_1707_03771_gb300 import binding, build
    build.build()
    return binding


def _system(waters, drop):
    """A water cluster without the last `drop` shells of its orbital basis (orders that are not multiples of 10)."""
    s = clusters.water_cluster(waters, 40 + waters)
    return clusters.System(atoms=s.atoms, basis=s.basis[:len(s.basis) - drop], aux=s.aux, label=f"{s.label}-{drop}")


@pytest.mark.parametrize("waters,drop", [(1, 0), (1, 1), (1, 2), (2, 0), (2, 3), (3, 0), (3, 2), (4, 0), (4, 3), (5, 0), (5, 1),
                                         (6, 0)])
def test_orbitals_of_a_converged_run(lib, waters, drop):
    system = _system(waters, drop)
    with lib.Handle(system) as h:
        r = h.scf(conv_E=1e-11, conv_err=1e-9)
        assert r["converged"] and r["n_dropped"] == 0
        F, S, C, eps = (h.matrix(k) for k in ("F", "S", "C", "eps"))
        again = h.scf(conv_E=1e-11, conv_err=1e-9)
    assert np.all(np.diff(eps) >= 0)
    assert np.abs(C.T @ S @ C - np.eye(h.n)).max() <= 1e-10
    assert np.abs(F @ C - S @ C * eps).max() <= 1e-7 * np.abs(C).max()
    assert again["energy"] == r["energy"] and again["iterations"] == r["iterations"]   # reproducible
