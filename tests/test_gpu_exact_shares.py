"""Population powers on wavelength tables whose shares span many powers of two: the
integer sums against the FP64 sums of the same library, which a zero written as
-0.0 selects for the block (the row's values stay the same).

Both sums are right to a few 1e-16 of each population's own power, and everything
after them is the same: ln T moves by a fifth of that, and a value e^{-x} off the
Wien side (x <= 25 where it still carries 1e-9 of the row) and the double-float
rounding of 1/T (2^-48) by x times as much, 1e-13 at most."""
import numpy as np
import pytest

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


def _run(S, a, lam, m, pair):
    import torch
    n = a.shape[0]
    d = lambda v, t: torch.as_tensor(np.ascontiguousarray(v), dtype=t, device="cuda")
    em = torch.full((n, S.NEMIT), float("nan"), dtype=torch.float64, device="cuda")
    if pair:  # the table under test as the second one, behind a field without power
        one = np.array([0.4, 0.7, 1.1])
        S.skirt_dust_emission_pair(d(np.zeros((n, 3)), torch.float64), n, one, d(a, torch.float64), lam,
                                   d(m, torch.float32), em)
    else:
        S.skirt_dust_emission(d(a, torch.float64), n, lam.size, lam, d(m, torch.float32), S.EMIT_EXACT, None, em)
    return em.cpu().numpy()


@pytest.mark.parametrize("pair", [False, True])
@pytest.mark.parametrize("n_in", [2, 100, 257])
@pytest.mark.parametrize("lo,hi", [(0.09, 10.0), (1.0, 1e3), (1.0, 1e6), (1.0, 1e9), (1e-9, 1e12), (1.0, 1e20)])
def test_integer_sums_against_fp64(S, lo, hi, n_in, pair):
    rng = np.random.default_rng(n_in)
    lam = np.geomspace(lo, hi, n_in)
    rows = []
    for j in sorted({0, 1, n_in // 2, n_in - 1}):           # one column holds the power
        rows.append(np.where(np.arange(n_in) == j, rng.uniform(0.5, 1.0), 0.0))
    for slope in (-1.0, 0.0, 0.7):                          # all columns do
        rows.append(lam ** slope / (lam ** slope).max() * rng.uniform(0.1, 1.0, n_in))
    rows.append(10.0 ** rng.uniform(-30.0, 0.0, n_in))      # few do
    a = np.repeat(np.array(rows), 4, axis=0)
    if n_in > 2:
        a[:, [5, min(n_in - 2, 255)]] = 0.0                 # the columns that select the form
    else:
        a = a[:4]                                           # the power in column 0
        a[:, 1] = 0.0
    # power per mass such that the populations lie at 3 K to 2000 K, apart by their shares
    m = (a.sum(axis=1) / np.tile([1e-2, 1e1, 1e4, 1e7], a.shape[0] // 4)).astype(np.float32)
    b = a.copy()
    b[:, [1] if n_in == 2 else [5, min(n_in - 2, 255)]] = -0.0
    if n_in == 257:
        b[:, 256] = np.where(b[:, 256] == 0.0, -0.0, b[:, 256])  # (a block of one column)
    got, want = _run(S, a, lam, m, pair), _run(S, b, lam, m, pair)
    assert np.all(np.isfinite(want)) and np.all(want.sum(axis=1) > 0)
    big = want > 1e-9 * want.sum(axis=1, keepdims=True)
    np.testing.assert_allclose(got[big], want[big], rtol=1e-12)
