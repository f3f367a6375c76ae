"""A rebuild of B while a Coulomb call on the old one is still queued: df_coulomb_noalloc returns without waiting, and
the handle may have been given another stream since. The rebuild takes over the old B's memory, so it has to wait for
those reads. A spin kernel of about a quarter of a second ahead of the Coulomb call keeps it from starting early."""
import ctypes

import numpy as np
import pytest

from paper_1707_03771_gb300 import clusters

pytestmark = pytest.mark.gpu

TOL = 1e-12   # relative to max |J|, as in the J/K kernel parity test


@pytest.mark.parametrize("keep", [False, True])
@pytest.mark.parametrize("whitening", ["FP64", "SPLIT"])
def test_rebuild_waits_for_a_queued_coulomb_call(keep, whitening):
    torch = pytest.importorskip("torch")
    from paper_1707_03771_gb300 import binding, build
    build.build()
    lib = binding.load()
    lib.df_set_stream.argtypes = [ctypes.c_void_p, ctypes.c_void_p]
    how = getattr(binding, f"DF_WHITEN_{whitening}")
    first, second = torch.cuda.Stream(), torch.cuda.Stream()
    with binding.Handle(clusters.workload("water2")) as h:
        h.build_B(keep_3c=keep, whitening=how)
        C = np.linalg.qr(np.random.default_rng(2).normal(size=(h.n, h.nocc)))[0]
        D = 2 * C @ C.T
        J_ref = h.jk(D, C)[0]
        dD = torch.from_numpy(D).cuda()
        dJ = torch.full_like(dD, float("nan"))
        torch.cuda.synchronize()
        assert lib.df_set_stream(h.h, first.cuda_stream) == 0
        with torch.cuda.stream(first):
            torch.cuda._sleep(500_000_000)
        h.coulomb_noalloc(dD.data_ptr(), dJ.data_ptr())
        assert lib.df_set_stream(h.h, second.cuda_stream) == 0
        h.build_B(keep_3c=keep, whitening=how)
        torch.cuda.synchronize()
        J = dJ.cpu().numpy()
        again = h.jk(D, C)[0]
        assert lib.df_set_stream(h.h, None) == 0
    assert np.abs(J - J_ref).max() <= TOL * np.abs(J_ref).max()
    assert np.array_equal(again, J_ref)
