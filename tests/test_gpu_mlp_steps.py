"""The network's step kernel at the edges of its tiles (16 x 16 outputs, 128 contraction elements, 256 inputs an
update task): gradients and the FP32 forward pass against the FP64 oracle, and several Adam steps.

Tolerances. A sum of k FP32 products is off by at most k eps sum|a b|; through the layers that gives at most
1e-4 of the largest gradient at these sizes (the bound of the gradient test at smaller ones). An Adam update moves
a parameter by lr g / (|g| + eps) at first, and by a smooth function of the same gradients later, so a relative
error of 1e-2 in a gradient above a hundredth of the largest changes it by less than 2e-2 lr a step. Rows are copies
of one sample where the order of a batch's rows must not matter."""
import numpy as np
import pytest

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_1707_03771_gb300 import binding, build
    build.build()
    return binding


def _net(lib, dims, seed):
    net = lib.Mlp(dims[0], dims[1], len(dims) - 2, dims[-1], seed=seed)
    p = net.params() + (np.random.default_rng(seed).normal(size=net.nparams) * 0.02).astype(np.float32)
    net.set_params(p)
    return net, p


@pytest.mark.parametrize("dims", [[1, 1, 1], [57, 16, 16, 17], [128, 129, 31], [300, 260, 260, 15], [26, 64, 300]])
@pytest.mark.parametrize("rows", [1, 16, 17, 70])
def test_gradients_and_forward_on_ragged_shapes(lib, dims, rows):
    net, p = _net(lib, dims, 3)
    rng = np.random.default_rng(rows)
    X = rng.normal(size=(rows, dims[0])).astype(np.float32)
    Y = rng.normal(size=(rows, dims[-1])).astype(np.float32)
    loss, g = net.gradients(X, Y)
    ref = omlp.gradient(p.astype(np.float64), dims, X.astype(np.float64), Y.astype(np.float64))
    ref_loss = omlp.loss(p.astype(np.float64), dims, X.astype(np.float64), Y.astype(np.float64))
    assert abs(loss - ref_loss) <= 1e-5 * abs(ref_loss)
    assert np.abs(g - ref).max() <= 1e-4 * np.abs(ref).max()
    # the loss of the predictions is the loss: the forward pass alone gives the same outputs
    pred = net.predict(X, bf16=False).astype(np.float64)
    assert abs(np.mean((pred - Y) ** 2) - ref_loss) <= 1e-5 * abs(ref_loss)
    net.close()


@pytest.mark.parametrize("dims,rows", [([5, 17, 19], 1), ([57, 48, 48, 33], 17), ([26, 300, 40], 16)])
def test_adam_steps(lib, dims, rows):
    net, p = _net(lib, dims, 7)
    rng = np.random.default_rng(1)
    X = np.repeat(rng.normal(size=(1, dims[0])), rows, axis=0).astype(np.float32)
    Y = np.repeat(rng.normal(size=(1, dims[-1])), rows, axis=0).astype(np.float32)
    lr, steps = 1e-3, 3
    hist = net.train(X, Y, epochs=steps, batch=rows, lr=lr, seed=1)
    q, m, v, big = p.astype(np.float64), 0.0, 0.0, None
    for t in range(1, steps + 1):
        ref_loss = omlp.loss(q, dims, X.astype(np.float64), Y.astype(np.float64))
        assert abs(hist[t - 1] - ref_loss) <= 1e-3 * ref_loss
        g = omlp.gradient(q, dims, X.astype(np.float64), Y.astype(np.float64))
        big = (np.abs(g) > 1e-2 * np.abs(g).max()) & (True if big is None else big)
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        q = q - lr * (m / (1 - 0.9 ** t)) / (np.sqrt(v / (1 - 0.999 ** t)) + 1e-8)
    got = net.params()
    assert big.sum() > 0
    assert np.abs(got - q)[big].max() <= 2e-2 * lr * steps
    net.close()
