"""The tensor-core exchange over every tile width and over column counts that do not fill their tiles (the last
tile of Y is narrower, zero 16-blocks of the contraction take no product): the same bits for every width, and K
within the splitting's own error bound of the FP64 K.

Bound. With S slices of 7 bits, a value of a row scaled by 2^e is represented to 2^(e - 7S - 1), and the dropped
slice pairs (s + t > S + 1) of a product add at most (S - 1) 2^12 2^(-7 (S + 2)) of both scales: per term of a
contraction at most 2^(e_a + e_b - 7S) (1 + (S - 1) / 4). Y sums n such terms, K naux ldy of them over Y's slices
plus twice |Y| times Y's own error."""
import os

import numpy as np
import pytest

from paper_1707_03771_gb300 import clusters

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def handle():
    from paper_1707_03771_gb300 import binding, build
    build.build()
    with binding.Handle(clusters.water_cluster(3, 9)) as h:
        h.build_B()
        yield binding, h, h.rows(1, 0, h.naux)


def _scale(a, axis):
    """The power of two above max |a| along axis."""
    m = np.abs(a).max(axis=axis)
    return np.where(m > 0, 2.0 ** np.ceil(np.log2(np.maximum(m, 1e-300) * (1 + 1e-12))), 0.0)


@pytest.mark.parametrize("packed", ["0", "1"])
@pytest.mark.parametrize("nocc", [1, 16, 17, 33, 48, 70, 81, 100, 129])
def test_exchange_over_tile_widths_and_column_counts(handle, nocc, packed):
    lib, h, B = handle
    rng = np.random.default_rng(nocc)
    C = rng.standard_normal((h.n, nocc)) / np.sqrt(h.n)
    D = 2 * C @ C.T
    K64 = h.jk(D, C, lib.DF_PREC_FP64)[1]
    Y = np.einsum("gmn,ni->gmi", B, C)
    ldy = (nocc + 31) // 32 * 32
    os.environ["DFHF_TC_PACKED"] = packed
    try:
        for S in (3, 5):
            per = 2.0 ** (-7 * S) * (1 + (S - 1) / 4)
            eB = _scale(B, 2) if packed == "0" else np.broadcast_to(_scale(B, (1, 2))[:, None], B.shape[:2])
            dY = h.n * per * eB[:, :, None] * _scale(C, 0)[None, None, :]
            eY = _scale(np.abs(Y) + dY, (0, 2))
            bound = h.naux * ldy * per * np.outer(eY, eY)
            cross = np.einsum("gmi,gni->mn", np.abs(Y) + dY, dY)
            bound = bound + cross + cross.T
            ref = None
            for tiles in ("32,32,2", "48,48,2", "64,64,2", "80,48,2"):
                os.environ["DFHF_TC_TILES"] = tiles
                K = h.jk(D, C, lib.DF_PREC_SPLIT, S)[1]
                assert np.all(np.abs(K - K64) <= bound), (S, tiles, np.abs(K - K64).max())
                assert np.array_equal(K, K.T)
                ref = K if ref is None else ref
                assert np.array_equal(K, ref), (S, tiles)
            # the autotuned choice, with its own split of the contraction
            del os.environ["DFHF_TC_TILES"]
            assert np.all(np.abs(h.jk(D, C, lib.DF_PREC_SPLIT, S)[1] - K64) <= bound)
    finally:
        os.environ.pop("DFHF_TC_TILES", None)
        os.environ.pop("DFHF_TC_PACKED", None)
