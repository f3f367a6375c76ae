"""The tile width that df_timings reports for the tensor-core Y kernel is that of the kernel that ran, forced or chosen
by the autotuner, over column counts on both sides of 48 and 64."""
import os
import re

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
        yield binding, h


def _y_widths(call):
    """The widths N of the kernels ozaki_tc_kernel<S, N, 0 or 3> that a call launches."""
    torch = pytest.importorskip("torch")
    from torch.profiler import ProfilerActivity, profile
    names = []
    for _ in range(2):                                        # a process's first profile may come back empty
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            call()
            torch.cuda.synchronize()
        names = names or [e.name for e in prof.events() if "ozaki_tc_kernel" in e.name]
    if not names:
        pytest.skip("no kernel records from the profiler")
    found = [re.search(r"ozaki_tc_kernel(?:<(\d+), (\d+), (\d+)>|ILi(\d+)ELi(\d+)ELi(\d+)E)", n) for n in names]
    found = [[int(x) for x in m.groups() if x is not None] for m in found]
    return {n for _, n, mode in found if mode in (0, 3)}


@pytest.mark.parametrize("packed", ["0", "1"])
@pytest.mark.parametrize("nocc", [15, 33, 48, 64, 81])
def test_reported_width_is_the_one_that_runs(handle, nocc, packed):
    lib, h = handle
    C = np.linalg.qr(np.random.default_rng(nocc).standard_normal((h.n, nocc)))[0]
    D = 2 * C @ C.T
    os.environ["DFHF_TC_PACKED"] = packed
    try:
        for S in (3, 5):
            for tiles in ("32", "48", "64", "80", None):
                if tiles:
                    os.environ["DFHF_TC_TILES"] = f"{tiles},48,2"
                else:
                    os.environ.pop("DFHF_TC_TILES", None)
                    h.jk(D, C, lib.DF_PREC_SPLIT, S)          # the autotuner's own launches come with the first call
                ran = _y_widths(lambda: h.jk(D, C, lib.DF_PREC_SPLIT, S))
                assert ran == {int(h.timings()["tc_y_tile_n"])}, (S, tiles)
                assert tiles is None or ran == {int(tiles)}
    finally:
        os.environ.pop("DFHF_TC_TILES", None)
        os.environ.pop("DFHF_TC_PACKED", None)
