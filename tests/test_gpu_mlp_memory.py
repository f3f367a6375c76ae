"""Training whose batches are large: the sample indices that a launch takes are bounded, whatever the number of steps.

60000 rows over 400 steps are 96 MB of indices as one launch; the largest launch holds 2^20 of them (4 MB). The host's
peak may grow by that, the samples and the allocator's rounding: 32 MB are allowed."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

SCRIPT = """
import resource
import numpy as np
from paper_1707_03771_gb300 import binding
peak = lambda: resource.getrusage(resource.RUSAGE_SELF).ru_maxrss / 1024
rng = np.random.default_rng(0)
X = rng.normal(size=(60000, 1)).astype(np.float32)
net = binding.Mlp(1, 1, 1, 1, seed=1)
net.train(X, X, epochs=1, batch=60000, lr=1e-3, seed=1)
before = peak()
net.train(X, X, epochs=400, batch=60000, lr=1e-3, seed=1)
print("GROWTH", peak() - before)
"""


def test_many_steps_of_large_batches_take_little_memory():
    from paper_1707_03771_gb300 import build
    build.build()
    out = subprocess.run([sys.executable, "-c", SCRIPT], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr[-2000:]
    assert float(out.stdout.split("GROWTH")[1]) < 32
