"""The dust source's cumulative distribution at the edges of its tiles (256
cells) and of its 32-wavelength columns: column sums, and packets drawn only
from the cells that emit, in proportion to their emission."""
import numpy as np
import pytest

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


def _grid(nxyz):
    nx, ny, nz = nxyz
    return W.Grid(nx, ny, nz, (0.0, float(nx), 0.0, float(ny), 0.0, float(nz)), np.zeros((nz, ny, nx), np.float32))


@pytest.mark.parametrize("nxyz", [(1, 1, 1), (31, 1, 1), (255, 1, 1), (256, 1, 1), (257, 1, 1), (64, 33, 9)])
@pytest.mark.parametrize("nl", [1, 31, 33, 100])
def test_column_sums(S, nxyz, nl):
    """In any order FP64 sums of n non-negative terms agree to n eps."""
    import torch
    g = S.Grid(_grid(nxyz))
    rng = np.random.default_rng(5)
    em = 10.0 ** rng.uniform(-12, 3, (g.ncell, nl)) * (rng.random((g.ncell, nl)) < 0.5)
    tot = S.skirt_emission_totals(g.h, torch.as_tensor(em, device="cuda"), nl)
    np.testing.assert_allclose(tot, em.sum(axis=0), rtol=2 * g.ncell * 2.3e-16, atol=0)
    for bad in (-1.0, np.nan, np.inf):
        e = torch.as_tensor(em, device="cuda").clone()
        e[-1, -1] = bad
        with pytest.raises(S.SkirtError):
            S.skirt_emission_totals(g.h, e, nl)
    g.close()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("cells", [(0,), (255, 256), (511,), (512, 700), (13, 300, 1023, 1049)])
def test_packets_start_in_the_emitting_cells(S, precision, cells):
    """Transparent grid of 1050 cells in a row: a packet's last position is its
    start.  The shares follow the emission within five binomial deviations."""
    import torch
    grid = _grid((1050, 1, 1))
    em = torch.zeros((1050, 2), dtype=torch.float64, device="cuda")
    w = np.arange(1, len(cells) + 1, dtype=np.float64) ** 2
    em[list(cells), 0] = torch.as_tensor(w, device="cuda")
    em[list(cells)[::-1], 1] = torch.as_tensor(w * 1e-300, device="cuda")
    n = 20000
    wl = W.Wavelengths(lam=np.array([1.0, 2.0]), kscale=np.ones(2), albedo=np.zeros(2), g=np.zeros(2), lsrc=None)
    prob = W.Problem("dust", grid, W.Source(W.SRC_DUST), wl, np.full(2, n, dtype=np.uint64), [], seed=9)
    rec = S.run_problem(prob, precision=precision, emission=em, nrec=n)["records"].cpu().numpy()
    for j in range(2):
        cell = np.floor(rec[j, :, 5]).astype(int)
        p = em[:, j].cpu().numpy()
        p = p / p.sum()
        assert np.all(p[cell] > 0)
        got = np.bincount(cell, minlength=1050) / n
        assert np.all(np.abs(got - p) <= 5 * np.sqrt(p * (1 - p) / n))
