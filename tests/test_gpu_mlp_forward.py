"""The FP32 forward pass on both sides of the row count from which it runs layer by layer in wide tiles: rows do not
depend on one another, and both kernels sum every element as one chain of multiply-adds, so the outputs of many rows
are those of the same rows in small groups, bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(1, 1, 1, 1), (57, 70, 3, 33), (26, 256, 1, 65), (130, 64, 2, 1)])
@pytest.mark.parametrize("rows", [1023, 1024, 1025, 2111])
def test_rows_do_not_depend_on_how_many_there_are(dims, rows):
    from paper_1707_03771_gb300 import binding, build
    build.build()
    rng = np.random.default_rng(rows)
    X = rng.normal(size=(rows, dims[0])).astype(np.float32)
    net = binding.Mlp(*dims, seed=4)
    net.set_params(net.params() + (rng.normal(size=net.nparams) * 0.02).astype(np.float32))
    whole = net.predict(X)
    parts = np.concatenate([net.predict(X[r:r + 300]) for r in range(0, rows, 300)])
    net.close()
    assert np.array_equal(whole, parts)
