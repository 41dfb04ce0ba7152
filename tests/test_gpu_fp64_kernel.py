"""The FP64 trace kernel at the edges of its crossing arithmetic, against the
oracle at the form's 1e-9: cells on either side of the deposit's series limit
(optical depth 1/16), paths longer than a round of crossings, very thick cells,
one-cell grids and every block size."""
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


def _compare(g, ref, n):
    a, b = g["records"].cpu().numpy(), ref["records"]
    assert np.array_equal(a[..., 0], b[..., 0])
    scale = np.abs(b[..., 1:]).max(axis=(0, 1))
    assert np.all(np.abs(a[..., 1:] - b[..., 1:]) <= 1e-9 * (np.abs(b[..., 1:]) + scale))
    np.testing.assert_allclose(g["absorbed"].cpu().numpy(), ref["absorbed"], rtol=1e-9, atol=1e-9 * ref["absorbed"].max())
    np.testing.assert_allclose(g["sed"].cpu().numpy(), ref["sed"], rtol=1e-9)


@pytest.mark.parametrize("tau_cell", [1e-12, 1e-4, 0.0624, 0.0626, 0.5, 40.0])
@pytest.mark.parametrize("n", [1, 23, 50])
def test_cell_optical_depths(S, oracle_lib, tau_cell, n):
    grid = W.uniform_grid(n, kr=tau_cell * n / 2.0)
    prob = W.Problem("cell", grid, W.Source(W.SRC_POINT, (0.1, -0.2, 0.3)), W.single_wavelength(albedo=0.3),
                     np.array([200], dtype=np.uint64), [W.Instrument(100.0, 50.0, 20.0, 2.0, 16)], seed=5)
    ref = oracle_lib.trace(prob, nrec=200)
    _compare(S.run_problem(prob, precision=S.PREC_FP64, nrec=200), ref, 200)


@pytest.mark.parametrize("block", [32, 256, 512])
@pytest.mark.parametrize("schedule", [0, 1])
def test_blocks_and_schedules(S, oracle_lib, block, schedule):
    prob = W.disk_problem(150, n=40, nlambda=3, npx=32, seed=2)
    ref = oracle_lib.trace(prob, nrec=150)
    _compare(S.run_problem(prob, precision=S.PREC_FP64, schedule=schedule, block=block, nrec=150), ref, 150)
