"""The exact solve's population powers (64-bit integer sums over blocks of 256
columns, FP64 for the blocks those cannot take) and its row batches, at their
edges, against the FP64 oracle: values that carry a row's energy to 1e-9, row
sums to 1e-12 (the bounds of the solve itself)."""
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


def _run(S, a, lam, m):
    import torch
    n = a.shape[0]
    em = torch.full((n, S.NEMIT), float("nan"), dtype=torch.float64, device="cuda")
    T = torch.full((n, 3), float("nan"), dtype=torch.float32, device="cuda")
    S.skirt_dust_emission(torch.as_tensor(a, dtype=torch.float64, device="cuda"), n, lam.size, lam,
                          torch.as_tensor(m, dtype=torch.float32, device="cuda"), S.EMIT_EXACT, None, em, T)
    return em.cpu().numpy(), T.cpu().numpy()


def _check(em, T, a, lam, m):
    # rows whose power is near the smallest normal number: the reference in units of
    # 2^-600 (power and mass alike, which leaves the temperatures), where its own
    # products do not underflow
    u = np.where(np.abs(a).max(axis=1) < 1e-200, 2.0 ** 600, 1.0)
    ref, Tr, _ = E.exact_emission(a * u[:, None], lam, m.astype(np.float64) * u)
    ref = ref / u[:, None]
    big = ref > 1e-9 * ref.sum(axis=1, keepdims=True)
    np.testing.assert_allclose(em[big], ref[big], rtol=1e-9)
    np.testing.assert_allclose(em.sum(axis=1), ref.sum(axis=1), rtol=1e-12)
    np.testing.assert_allclose(T, Tr, rtol=1e-6)


@pytest.mark.parametrize("n_in", [1, 2, 31, 33, 255, 256, 257, 513, 800])
def test_column_blocks(S, n_in):
    lam = np.geomspace(0.09, 10.0, n_in) if n_in > 1 else np.array([0.5])
    a, m = W.absorbed_spectra(57, lam, seed=n_in)
    a[0] = 0.0                                   # no power
    a[1, :] = 0.0
    a[1, -1] = m[1]                              # a single entry, in the last column
    a[2] *= 10.0 ** np.linspace(-280, 0, n_in)   # a wide range within the row
    a[3] = m[3] * np.nextafter(1.0, 0.0) / n_in  # all entries alike, every significand bit set
    a[4, ::2] = 0.0
    em, T = _run(S, a, lam, m)
    _check(em, T, a, lam, m)


def test_blocks_that_integers_cannot_take(S):
    """Negative entries, and rows whose entries are all tiny, are summed in FP64
    (a negative entry only lowers a population's power; a row with a NaN or an
    infinity gives neither a zero row nor disturbs its neighbours)."""
    lam = np.geomspace(0.09, 10.0, 300)
    a, m = W.absorbed_spectra(40, lam, seed=2)
    a[0, 7] = -1e-3 * a[0].sum()
    a[1, 280] = -1e-3 * a[1].sum()               # in the second block
    a[2, 5] = -0.0
    a[3] *= 1e-300
    m[3] = 1e-30
    a[4, 100] = np.nan
    a[5, 100] = np.inf
    ok = np.setdiff1d(np.arange(40), [4, 5])
    em, T = _run(S, a, lam, m)
    _check(em[ok], T[ok], a[ok], lam, m[ok])
    assert not np.any(em[4] > 0)                 # no power comes of a NaN


@pytest.mark.parametrize("n", [1, 9, 3648, 3649, 10944, 40000])
def test_row_batches(S, n):
    lam = np.geomspace(0.09, 10.0, 24)
    a, m = W.absorbed_spectra(n, lam, seed=4)
    em, T = _run(S, a, lam, m)
    pick = np.unique(np.concatenate([np.arange(min(n, 25)), np.arange(max(0, n - 25), n)]))
    _check(em[pick], T[pick], a[pick], lam, m[pick])
    np.testing.assert_allclose(em.sum(axis=1), a.sum(axis=1), rtol=1e-12)
