"""Every parameter of a training step takes the learning rate and the bias
corrections of that step, in batches of so many tiles that the blocks of the
gradient sum start one after the other.

The batch is the whole data, so every epoch is one step over all rows (in another
order), and the reference is the network's own gradient followed by Adam in numpy.
The bound is on the whole change of each block of 128 parameters (one block of the
sum): Adam divides a gradient's noise out of no parameter, so a block that took
another step's rate (they fall from 1 to 0.05 of the first over the run) would be
off by tens of per cent, while sums in another order, and the BF16 weights that
follow from them, move a block's norm by well under one."""
import math

import numpy as np
import pytest

from oracle import emission as E
from paper_1705_04702_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1705_04702_gb300 import build
    build.build()
    from paper_1705_04702_gb300 import skirt
    return skirt


@pytest.mark.parametrize("rows,steps", [(4096, 5), (16384, 4)])
def test_blocks_take_their_own_step(S, rows, steps):
    import torch
    lam = np.geomspace(0.09, 10.0, 40)
    a, m = W.absorbed_spectra(rows, lam, seed=6)
    _, x, _ = E.band_features(a, lam, m.astype(np.float64))
    x = x.astype(np.float32)
    lab = np.exp(-0.5 * ((np.arange(100)[None, :] - 30.0 - 40.0 * np.random.default_rng(1).random((rows, 1))) / 9.0) ** 2)
    lr, b1, b2, eps = np.float32(2e-3), 0.9, 0.999, 1e-8

    net = S.MLP(seed=5)
    start = net.get_params()[0].astype(np.float64)
    net.train(torch.as_tensor(x, device="cuda"), torch.as_tensor(lab, device="cuda"), rows, epochs=steps, batch=rows, lr=lr)
    got, mean, std, _, _ = net.get_params()
    net.close()

    ref = S.MLP(seed=5)
    p = start.copy()
    t = torch.as_tensor((lab / lab.sum(axis=1, keepdims=True)).astype(np.float32), device="cuda")
    xs = torch.as_tensor((x - mean) / std, device="cuda")
    m1, m2 = np.zeros_like(p), np.zeros_like(p)
    for k in range(steps):
        ref.set_params(p.astype(np.float32))
        g = ref.grad(xs, t, rows)[0].astype(np.float64)
        m1 = b1 * m1 + (1 - b1) * g
        m2 = b2 * m2 + (1 - b2) * g * g
        rate = lr * (0.05 + 0.95 * 0.5 * (1.0 + math.cos(math.pi * k / (steps - 1))))
        p -= rate * (m1 / (1 - b1 ** (k + 1))) / (np.sqrt(m2 / (1 - b2 ** (k + 1))) + eps)
    ref.close()
    for i in range(0, p.size, 128):
        want, have = p[i:i + 128] - start[i:i + 128], got[i:i + 128] - start[i:i + 128]
        assert np.linalg.norm(have - want) <= 0.05 * np.linalg.norm(want), i // 128
