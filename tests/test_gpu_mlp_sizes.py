"""Gradient and training steps of the chemical-potential network at the edges of a block's 16 samples and of the
grid (608 blocks, several groups of samples each beyond 9728), and the memory a call takes.

Tolerances.  Gradient: every entry is an FP32 sum over the samples of products of four or five rounded factors
(sums of 64 terms, tanhf): about 100 u = 6e-6 of the sum of the samples' magnitudes, 1e-5 allowed, as the other
test of the same kernel does.  Training: a step moves a parameter by lr m / sqrt(v), at most lr / sqrt(1 - b2) / ... of
order lr; its relative error is that of the gradient, so entries whose gradient stays above 1e-2 of its samples'
magnitudes in every step (error below 1e-3) agree to 1e-2 lr per step."""
import threading

import numpy as np
import pytest

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu


def data(n, seed):
    rng = np.random.default_rng(seed)
    return rng.normal(0, 1, (n, 32)).astype(np.float32), rng.normal(0, 0.5, n).astype(np.float32)


def start(seed):
    import torch
    import paper_1005_0088_gb300 as nd
    P = torch.zeros(nd.NDSI_MLP_PARAMS, dtype=torch.float32, device="cuda")
    nd.ndsi_mlp_init(P, seed)
    return nd, torch, P


def magnitudes(theta, X, T):
    """Sum over the samples of the gradient terms' magnitudes, over n (vectorised over the samples)."""
    p = omlp.unpack(theta)
    y, (X, h1, h2) = omlp.forward(theta, X)
    dy = np.abs(2.0 * (y - T) / len(T))
    dz2 = np.outer(dy, np.abs(p["W3"])) * (1.0 - h2 ** 2)
    dz1 = (dz2 @ np.abs(p["W2"])) * (1.0 - h1 ** 2)
    return omlp.pack({"W3": np.abs(h2).T @ dy, "b3": [dy.sum()], "W2": dz2.T @ np.abs(h1), "b2": dz2.sum(0),
                      "W1": dz1.T @ np.abs(X), "b1": dz1.sum(0)})


@pytest.mark.parametrize("n", [1, 15, 16, 17, 9727, 9728, 9729, 20007])
def test_gradient(n):
    nd, torch, P = start(3)
    X, T = data(n, n)
    G = torch.zeros_like(P)
    L = torch.zeros(1, dtype=torch.float32, device="cuda")
    nd.ndsi_mlp_grad(P, torch.as_tensor(X, device="cuda"), torch.as_tensor(T, device="cuda"), n, G, L)
    theta = P.cpu().numpy().astype(np.float64)
    X, T = X.astype(np.float64), T.astype(np.float64)
    ref, mag = omlp.grad(theta, X, T), magnitudes(theta, X, T)
    bad = np.abs(G.cpu().numpy() - ref) > 1e-5 * mag + 1e-12
    assert not bad.any(), np.nonzero(bad)[0][:10]
    assert abs(float(L.cpu()[0]) - omlp.loss(theta, X, T)) < 1e-5 * omlp.loss(theta, X, T)


@pytest.mark.parametrize("n", [1, 15, 16, 17, 9729])
def test_training_steps_are_adam(n):
    nd, torch, P = start(11)
    X, T = data(n, 100 + n)
    lr, steps = 1e-3, 3
    theta = P.cpu().numpy().astype(np.float64)
    loss = nd.ndsi_mlp_train(P, torch.as_tensor(X, device="cuda"), torch.as_tensor(T, device="cuda"), n, steps, lr)
    X, T = X.astype(np.float64), T.astype(np.float64)
    b1, b2, eps = 0.9, 0.999, 1e-8
    m, v = np.zeros_like(theta), np.zeros_like(theta)
    firm = np.ones(theta.size, bool)
    for s in range(1, steps + 1):
        g = omlp.grad(theta, X, T)
        firm &= np.abs(g) > np.maximum(1e-2 * magnitudes(theta, X, T), 1e-5)
        last = omlp.loss(theta, X, T)
        m = b1 * m + (1 - b1) * g
        v = b2 * v + (1 - b2) * g * g
        theta = theta - lr * (m / (1 - b1 ** s)) / (np.sqrt(v / (1 - b2 ** s)) + eps)
    assert firm.mean() > 0.5
    diff = np.abs(P.cpu().numpy() - theta)
    assert diff[firm].max() < 1e-2 * lr * steps
    assert diff.max() < 2.01 * lr * steps * 2          # no entry moves further than its steps allow
    assert abs(loss - last) < 1e-4 * max(last, 1e-3)


def test_scratch_does_not_grow_with_the_samples():
    nd, torch, P = start(5)
    n = 1 << 21
    X = torch.randn(n, 32, device="cuda") * 0.5
    T = torch.randn(n, device="cuda") * 0.5
    nd.ndsi_mlp_train(P, X[:1024].contiguous(), T[:1024].contiguous(), 1024, 1, 1e-3)   # loads the kernels
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    done, seen = threading.Event(), []

    def watch():
        while not done.is_set():
            seen.append(torch.cuda.mem_get_info()[0])

    w = threading.Thread(target=watch)
    w.start()
    nd.ndsi_mlp_train(P, X, T, n, 40, 1e-3)
    done.set()
    w.join()
    assert len(seen) >= 3
    assert before - min(seen) <= 64 << 20, (before - min(seen)) >> 20
