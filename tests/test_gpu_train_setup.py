"""What training derives from its rows: the guard (a quantile of the rows' dominant-
band share, selected on the device) and the features' statistics, against numpy;
and steps on batches whose tiles are not full or whose partial sums fill several
chunks."""
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


@pytest.mark.parametrize("n,q", [(32, 0.5), (33, 0.99), (1000, 0.01), (1000, 0.999), (20001, 0.99)])
def test_guard_and_statistics(S, n, q):
    import torch
    rng = np.random.default_rng(n)
    f = rng.normal(-5.0, 2.0, (n, 32)).astype(np.float32)
    f[1] = f[0]                                   # equal shares
    f[2, 3] = 10.0                                # a share of one
    em = rng.random((n, 100))
    net = S.MLP(seed=2)
    net.train(torch.as_tensor(f, device="cuda"), torch.as_tensor(em, dtype=torch.float64, device="cuda"), n, epochs=1,
              batch=32, guard_quantile=q)
    share = np.sort(E.dominant_share(f))
    k = int(np.float32(q) * np.float64(n - 1))
    # FP32 sums of 32 exponentials on the device: a few ulp
    np.testing.assert_allclose(net.get_guard(), share[k], rtol=3e-6)
    _, mean, std, lo, hi = net.get_params()
    np.testing.assert_allclose(mean, f.astype(np.float64).mean(axis=0), rtol=1e-6)
    np.testing.assert_allclose(std, f.astype(np.float64).std(axis=0), rtol=1e-5)
    np.testing.assert_array_equal(lo, f.min(axis=0))
    np.testing.assert_array_equal(hi, f.max(axis=0))
    net.close()


@pytest.mark.parametrize("batch", [32, 33, 100, 2048, 2080, 4100])
def test_steps_of_every_batch_shape(S, batch):
    """Ten steps on labels that do not depend on the features lower the mean
    cross-entropy towards the labels' entropy and repeat bit for bit."""
    import torch
    n = batch * 10
    lam = np.geomspace(0.09, 10.0, 40)
    a, m = W.absorbed_spectra(n, lam, seed=1)
    _, x, _ = E.band_features(a, lam, m.astype(np.float64))
    lab = np.tile(np.exp(-0.5 * ((np.arange(100) - 40.0) / 9.0) ** 2), (n, 1))
    out = []
    for _ in range(2):
        net = S.MLP(seed=3)
        h = net.train(torch.as_tensor(x, dtype=torch.float32, device="cuda"),
                      torch.as_tensor(lab, dtype=torch.float64, device="cuda"), n, epochs=3, batch=batch)
        out.append((h.copy(), net.get_params()[0].copy()))
        net.close()
    assert np.all(np.diff(out[0][0]) < 0)
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
