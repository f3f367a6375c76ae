"""Orbitals of an FP64 run that does not converge, after many iterations: as orthonormal as after two.

With C = X V^T, C^T S C - 1 = V (X^T S X - 1) V^T + V V^T - 1. The first part has one spectral norm for every run on a
molecule, the second that of the eigenvectors. Dot products of n terms round to sqrt(n) eps as a rule, a matrix of such
errors has the norm 2 n eps, which is allowed twice for either run, with a factor of two for what the matrix products
here add."""
import numpy as np
import pytest

from paper_1707_03771_gb300 import clusters

pytestmark = pytest.mark.gpu


def _stretched(waters, factor):
    """Waters whose O-H bonds are `factor` times as long, where a small DIIS space oscillates."""
    atoms = clusters.water_cluster(waters, 5).atoms.copy()
    xyz = atoms["xyz"].copy()
    for o in range(0, len(atoms), 3):
        xyz[o + 1:o + 3] = xyz[o] + factor * (xyz[o + 1:o + 3] - xyz[o])
    atoms["xyz"] = xyz
    return clusters.make_system(atoms)


@pytest.mark.parametrize("waters", [1, 2])
def test_orthonormality_does_not_drift(waters):
    from paper_1707_03771_gb300 import binding, build
    build.build()
    norms = []
    for iterations in (2, 400):
        with binding.Handle(_stretched(waters, 3.0)) as h:
            r = h.scf(conv_E=1e-300, conv_err=1e-300, max_iter=iterations, diis_size=2)
            assert not r["converged"]
            C, S, n = h.matrix("C"), h.matrix("S"), h.n
        norms.append(np.linalg.norm(C.T @ S @ C - np.eye(n), 2))
    assert norms[1] <= norms[0] + 8 * n * 2.0 ** -53
