"""The triangular solve of one diagonal block (up to 64 rows), whose quotients come from a reciprocal and two residual
corrections: every bit is that of forward substitution with fused multiply-adds and IEEE divisions, row by row."""
import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <cmath>
extern "C" void solve(const double* L, int m, double* Z, int n) {
    for (int j = 0; j < n; ++j)
        for (int i = 0; i < m; ++i) {
            double t = Z[i * n + j];
            for (int k = 0; k < i; ++k) t = fma(-L[i * m + k], Z[k * n + j], t);
            Z[i * n + j] = t / L[i * m + i];
        }
}
"""


@pytest.mark.parametrize("m,n", [(1, 1), (7, 33), (63, 40), (64, 1000)])
@pytest.mark.parametrize("spread", [1.0, 1e6])
def test_bits_of_forward_substitution(tmp_path, m, n, spread):
    torch = pytest.importorskip("torch")
    from paper_1707_03771_gb300 import binding, build
    build.build()
    (tmp_path / "ref.cpp").write_text(SOURCE)
    so = str(tmp_path / "ref.so")
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-o", so, str(tmp_path / "ref.cpp")], check=True)
    rng = np.random.default_rng(m + n)
    L = np.tril(rng.normal(size=(m, m)) / np.sqrt(m), -1) + np.diag(np.exp(rng.uniform(-np.log(spread), 0.7, m)))
    Z = rng.normal(size=(m, n))
    dL, dZ = torch.from_numpy(L).cuda(), torch.from_numpy(Z).cuda()
    fn = binding.load()._ZN4dfhf15tri_solve_lowerEP11CUstream_stPKdixPdix
    fn.restype = None
    fn.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int, ctypes.c_longlong, ctypes.c_void_p, ctypes.c_int,
                   ctypes.c_longlong]
    fn(torch.cuda.current_stream().cuda_stream, dL.data_ptr(), m, m, dZ.data_ptr(), n, n)
    torch.cuda.synchronize()
    ptr = ctypes.POINTER(ctypes.c_double)
    ctypes.CDLL(so).solve(L.ctypes.data_as(ptr), m, Z.ctypes.data_as(ptr), n)
    assert np.array_equal(dZ.cpu().numpy(), Z)
