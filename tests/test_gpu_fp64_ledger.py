"""The FP64 form's ledger counts what the cells took: `absorbed` is the sum of the
deposits, not what the path's optical depth says they should add up to, so that a
deposit that goes missing shows in the ledger's balance."""
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


def test_deposits_that_underflow_are_not_absorbed(S):
    """60 cells of optical depth 1e-4 and a packet of 1e-320: a deposit would be a
    fifth of the smallest number and is zero, the path's share of it is 12."""
    n = 60
    grid = W.Grid(n, 1, 1, (-1.0, 1.0, -1.0, 1.0, -1.0, 1.0), np.full((1, 1, n), 1e-4 * n / 2.0, dtype=np.float32))
    prob = W.Problem("beam", grid, W.Source(W.SRC_BEAM, (-1.0, 0.0, 0.0), (1.0, 0.0, 0.0)),
                     W.single_wavelength(albedo=0.0, lsrc=1e-320), np.array([1], dtype=np.uint64), [], seed=1)
    r = S.run_problem(prob, precision=S.PREC_FP64)
    assert r["ledger"]["emitted"] == 1e-320
    assert float(r["absorbed"].sum()) == 0.0 and r["ledger"]["absorbed"] == 0.0


@pytest.mark.parametrize("octree", [False, True])
def test_ledger_is_the_table(S, octree):
    """Both are sums of the same numbers in another order: 2e6 positive terms at most,
    whose rounding errors (2^-53 each, of either sign) stay far below 1e-12 of the sum."""
    if octree:
        tree = W.refine_octree(W.disk_density(), (-24.0, 24.0, -24.0, 24.0, -24.0, 24.0), 5, 2, 2e-3)
        prob = W.octree_problem(tree, 2000, npx=16)
    else:
        prob = W.torus_problem(n=32, nlambda=4, packet_scale=5e-5, npx=16)
    r = S.run_problem(prob, precision=S.PREC_FP64)
    table = r["absorbed"].sum(dim=0).cpu().numpy()
    np.testing.assert_allclose(np.asarray(r["ledger_per_lambda"])[:, 1], table, rtol=1e-12)
