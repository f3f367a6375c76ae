"""The network's step kernel against the same sums and updates done one by one on the host: equal in every bit.

The reference takes every element's products in ascending order of the contraction by fused multiply-adds in FP32,
divides and takes roots as IEEE 754 has it, and shuffles as the library does (std::shuffle, std::mt19937_64). The
shapes take the paths of the kernel's staging: contractions within and beyond one stage (768 to 1280 elements, whole
and ragged last stages), rows that are and are not multiples of four floats, tiles of every width (2 to 16 columns, by
the number of tiles), batches of more rows than a thread block has threads, weight updates over several stages of 64
rows, more steps than the bias corrections need to reach the largest FP32 below 1, and more than one launch."""
import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <algorithm>
#include <cmath>
#include <random>
#include <vector>
struct Net {
    int L;
    const int* d;
    const float* p;
    std::vector<std::vector<float>> Z, A, dZ;
    std::vector<size_t> w, b;
    Net(int layers, const int* dims, const float* params, int rows) : L(layers), d(dims), p(params) {
        size_t at = 0;
        for (int l = 0; l < L; ++l) {
            w.push_back(at);
            at += (size_t)d[l] * d[l + 1];
            b.push_back(at);
            at += d[l + 1];
            Z.emplace_back((size_t)rows * d[l + 1]);
        }
        A = dZ = Z;
    }
    void forward(const std::vector<const float*>& x) {
        for (int l = 0; l < L; ++l)
            for (size_t r = 0; r < x.size(); ++r) {
                const float* in = l == 0 ? x[r] : &A[l - 1][r * d[l]];
                for (int o = 0; o < d[l + 1]; ++o) {
                    float s = 0.f;
                    for (int k = 0; k < d[l]; ++k) s = fmaf(in[k], p[w[l] + (size_t)o * d[l] + k], s);
                    const float z = s + p[b[l] + o];
                    Z[l][r * d[l + 1] + o] = z;
                    A[l][r * d[l + 1] + o] = l < L - 1 ? fmaxf(z, 0.f) : z;
                }
            }
    }
    void gradient(const std::vector<const float*>& x, const std::vector<const float*>& y, float* g) {
        const int no = d[L], rows = (int)x.size();
        const float scale = 1.f / (float)((long long)rows * no);
        forward(x);
        for (int r = 0; r < rows; ++r)
            for (int o = 0; o < no; ++o) {
                const float e = A[L - 1][(size_t)r * no + o] - y[r][o];
                dZ[L - 1][(size_t)r * no + o] = 2.f * e * scale;
            }
        for (int l = L - 1; l >= 0; --l) {
            const int ni = d[l], n = d[l + 1];
            if (l > 0)
                for (int r = 0; r < rows; ++r)
                    for (int i = 0; i < ni; ++i) {
                        float s = 0.f;
                        for (int o = 0; o < n; ++o) s = fmaf(dZ[l][(size_t)r * n + o], p[w[l] + (size_t)o * ni + i], s);
                        dZ[l - 1][(size_t)r * ni + i] = Z[l - 1][(size_t)r * ni + i] <= 0.f ? 0.f : s;
                    }
            for (int o = 0; o < n; ++o) {
                float sb = 0.f;
                for (int r = 0; r < rows; ++r) sb += dZ[l][(size_t)r * n + o];
                g[b[l] + o] = sb;
                for (int i = 0; i < ni; ++i) {
                    float s = 0.f;
                    for (int r = 0; r < rows; ++r)
                        s = fmaf(dZ[l][(size_t)r * n + o], l == 0 ? x[r][i] : A[l - 1][(size_t)r * ni + i], s);
                    g[w[l] + (size_t)o * ni + i] = s;
                }
            }
        }
    }
};
extern "C" void gradient(int L, const int* d, const float* p, const float* X, const float* Y, int rows, float* out, float* g) {
    Net net(L, d, p, rows);
    std::vector<const float*> x, y;
    for (int r = 0; r < rows; ++r) {
        x.push_back(X + (size_t)r * d[0]);
        y.push_back(Y + (size_t)r * d[L]);
    }
    net.gradient(x, y, g);
    std::copy(net.A[L - 1].begin(), net.A[L - 1].end(), out);
}
extern "C" void train(int L, const int* d, float* p, long long np, const float* X, const float* Y, int ns, int epochs, int batch,
                      float lr, unsigned long long seed) {
    std::vector<float> g(np), m(np, 0.f), v(np, 0.f);
    std::vector<int> order(ns);
    for (int i = 0; i < ns; ++i) order[i] = i;
    std::mt19937_64 gen(seed);
    Net net(L, d, p, batch);
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    int t = 0;
    for (int ep = 0; ep < epochs; ++ep) {
        std::shuffle(order.begin(), order.end(), gen);
        for (int q = 0; q + batch <= ns; q += batch) {
            std::vector<const float*> x, y;
            for (int r = 0; r < batch; ++r) {
                x.push_back(X + (size_t)order[q + r] * d[0]);
                y.push_back(Y + (size_t)order[q + r] * d[L]);
            }
            net.gradient(x, y, g.data());
            ++t;
            const float c1 = 1.f - std::pow(b1, (float)t), c2 = 1.f - std::pow(b2, (float)t);
            for (long long i = 0; i < np; ++i) {
                m[i] = fmaf(1.f - b1, g[i], b1 * m[i]);
                v[i] = fmaf((1.f - b2) * g[i], g[i], b2 * v[i]);
                p[i] = p[i] - lr * (m[i] / c1) / (sqrtf(v[i] / c2) + eps);
            }
        }
    }
}
"""


@pytest.fixture(scope="module")
def lib():
    from paper_1707_03771_gb300 import binding, build
    build.build()
    return binding


@pytest.fixture(scope="module")
def ref(tmp_path_factory):
    d = tmp_path_factory.mktemp("mlp_ref")
    (d / "ref.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-o", str(d / "ref.so"), str(d / "ref.cpp")], check=True)
    return ctypes.CDLL(str(d / "ref.so"))


def _f(a):
    return a.ctypes.data_as(ctypes.POINTER(ctypes.c_float))


def _case(lib, dims, samples):
    """A network (nin, hidden, hidden layers, nout) with random biases, samples of its sizes, the layers' widths."""
    nin, nh, nl, nout = dims
    net = lib.Mlp(nin, nh, nl, nout, seed=3)
    rng = np.random.default_rng(samples + nin)
    net.set_params(net.params() + (rng.normal(size=net.nparams) * 0.02).astype(np.float32))
    X = rng.normal(size=(samples, nin)).astype(np.float32)
    Y = rng.normal(size=(samples, nout)).astype(np.float32)
    return net, X, Y, (ctypes.c_int * (nl + 2))(nin, *[nh] * nl, nout)


@pytest.mark.parametrize("dims", [(1, 1, 1, 1), (1281, 40, 1, 7), (1300, 9, 2, 1281), (3, 20, 1, 2500), (2564, 33, 1, 65)])
@pytest.mark.parametrize("rows", [5, 70, 300])
def test_gradients_bit_for_bit(lib, ref, dims, rows):
    net, X, Y, d = _case(lib, dims, rows)
    p, (_, g) = net.params(), net.gradients(X, Y)
    want, out = np.empty_like(g), np.empty((rows, dims[3]), np.float32)
    ref.gradient(dims[2] + 1, d, _f(p), _f(X), _f(Y), rows, _f(out), _f(want))
    assert np.array_equal(net.predict(X), out)
    assert np.array_equal(g, want)
    net.close()


@pytest.mark.parametrize("dims,samples,epochs,batch",
                         [((57, 48, 3, 33), 100, 6, 16), ((26, 20, 1, 30), 50, 120, 16), ((6, 300, 2, 9), 777, 3, 257),
                          ((40, 1030, 1, 17), 40, 3, 20), ((2, 3, 1, 2), 400000, 5, 400000)])
def test_training_bit_for_bit(lib, ref, dims, samples, epochs, batch):
    net, X, Y, d = _case(lib, dims, samples)
    want = net.params()
    net.train(X, Y, epochs, batch, 1e-3, seed=11)
    ref.train(dims[2] + 1, d, _f(want), ctypes.c_longlong(want.size), _f(X), _f(Y), samples, epochs, batch, ctypes.c_float(1e-3),
              ctypes.c_ulonglong(11))
    assert np.array_equal(net.params(), want)
    net.close()
