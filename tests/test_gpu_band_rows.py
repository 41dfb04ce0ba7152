"""Band compression with one band per lane at its edges, against the FP64
oracle (totals to 1e-13, features to a few FP32 ulp: the bounds of the step),
and against the row-per-lane form, which takes the same table at an address
that is not 16-byte aligned."""
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


def _run(S, a, lam, m, shift=0):
    import torch
    n, k = a.shape
    buf = torch.zeros(n * k + shift, dtype=torch.float64, device="cuda")
    buf[shift:] = torch.as_tensor(a, dtype=torch.float64).reshape(-1)
    f = torch.full((n, 32), float("nan"), dtype=torch.float32, device="cuda")
    t = torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")
    S.skirt_band_features(buf[shift:], n, k, lam, torch.as_tensor(m, dtype=torch.float32, device="cuda"), f, t)
    return f.cpu().numpy(), t.cpu().numpy()


@pytest.mark.parametrize("n_in", [1, 2, 3, 32, 33, 63, 128, 129, 200, 257, 500, 512])
@pytest.mark.parametrize("n", [1, 2, 31, 1000])
def test_sizes(S, n_in, n):
    lam = np.geomspace(0.09, 10.0, n_in) if n_in > 1 else np.array([0.5])
    a, m = W.absorbed_spectra(n, lam, seed=n_in + n)
    if n > 8:
        a[0] = 0.0
        m[1] = 0.0
        a[2] = 0.0
        a[2, n_in // 2] = m[2]
        a[3] *= 10.0 ** np.linspace(-290, 0, n_in)
        a[4] = np.nextafter(1.0, 0.0) * m[4]         # every significand bit set, all bands alike
        a[5, ::2] = 0.0
    f, t = _run(S, a, lam, m)
    _, x, total = E.band_features(a, lam, m.astype(np.float64))
    np.testing.assert_allclose(t, total, rtol=1e-13, atol=0)
    np.testing.assert_allclose(f, x, rtol=3e-7, atol=1e-6)
    # the other form: the same sums in FP64, so the same features but where an FP64
    # rounding error straddles an FP32 step (one ulp of the band sum)
    f2, t2 = _run(S, a, lam, m, shift=1)
    np.testing.assert_allclose(t, t2, rtol=1e-13, atol=0)
    np.testing.assert_allclose(f, f2, rtol=1.2e-7, atol=1e-7)


def test_uneven_bands_and_rows_for_fp64(S):
    """A linear wavelength grid (bands of 0 to over 16 columns: the row-per-lane
    form), one with up to 12 columns, and rows with negative, NaN, infinite, huge
    and tiny entries, which give what the row-per-lane form gives bit for bit."""
    for lam in (np.linspace(0.1, 10.0, 200), np.geomspace(0.1, 1.0, 256)):
        a, m = W.absorbed_spectra(100, lam, seed=8)
        f, t = _run(S, a, lam, m)
        _, x, total = E.band_features(a, lam, m.astype(np.float64))
        np.testing.assert_allclose(t, total, rtol=1e-13, atol=0)
        np.testing.assert_allclose(f, x, rtol=3e-7, atol=1e-6)
    lam = np.geomspace(0.09, 10.0, 200)
    a, m = W.absorbed_spectra(9, lam, seed=3)
    a[0, 3] = -1e-3 * a[0].sum()
    a[1, 100] = np.nan
    a[2, 199] = np.inf
    a[3] = 1e308
    a[4] = 1e-310
    a[5] = 0.0
    a[5, 7] = -0.0
    a[6, 50] = -np.inf
    f, t = _run(S, a, lam, m)
    f2, t2 = _run(S, a, lam, m, shift=1)
    np.testing.assert_array_equal(f[:7], f2[:7])
    np.testing.assert_array_equal(t[:7], t2[:7])
