"""df_mp2's peak of device memory: the pair integrals' rows take the room of the half-transformed B, which nothing reads
by then. All but the stated peak and 24 MB (the small arrays and the allocator's 2 MB blocks) of the free memory is taken
away before the call; with both arrays held it would need another 54 MB here."""
import numpy as np
import pytest

from paper_1707_03771_gb300 import clusters

pytestmark = pytest.mark.gpu


def test_peak_of_device_memory():
    torch = pytest.importorskip("torch")
    from paper_1707_03771_gb300 import binding, build
    build.build()
    nocc = 20
    with binding.Handle(clusters.water_cluster(12, 3)) as h:
        h.build_B()
        nvir = h.n - nocc
        C = np.linalg.qr(np.random.default_rng(1).normal(size=(h.n, h.n)))[0]
        eps = np.concatenate([np.linspace(-2, -0.5, nocc), np.linspace(0.1, 4, nvir)])
        ref = h.mp2(C, eps, nocc)
        torch.cuda.synchronize()
        tiles = (nvir + 31) // 32
        peak = 8 * nocc * (h.naux * nvir + max(h.naux * h.n, nvir * nvir + (nocc + 1) // 2 * tiles * (tiles + 1) // 2))
        ballast = torch.empty(torch.cuda.mem_get_info()[0] - peak - (24 << 20), dtype=torch.uint8, device="cuda")
        try:
            assert h.mp2(C, eps, nocc) == ref
        finally:
            del ballast
            torch.cuda.empty_cache()
