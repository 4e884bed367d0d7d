"""Threads that share a network: losses and gradients of batches of different sizes, which grow
and give back the network's workspace, are those of one call after the other, bit for bit."""
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

import paper_1912_08445_gb300 as mg

pytestmark = pytest.mark.gpu


def test_losses_of_threads():
    rng = np.random.default_rng(5)
    n_out = 12
    net = mg.MLP(n_out, seed=1)
    net.set_normalisation(np.zeros(4, np.float32), np.ones(4, np.float32))
    data = [(rng.normal(size=(n, 4)).astype(np.float32), rng.dirichlet(np.ones(n_out), size=n).astype(np.float32))
            for n in (64, 5000, 700, 130000, 64, 20000, 3, 90000)]      # (130000 rows: 295 MB of partial sums)
    want = [net.loss_grad(X, Y) for X, Y in data]
    with ThreadPoolExecutor(4) as ex:
        got = list(ex.map(lambda d: net.loss_grad(*d), data * 4))
    for k, (loss, grad) in enumerate(got):
        ref = want[k % len(data)]
        assert loss == ref[0] and np.array_equal(grad, ref[1]), k
