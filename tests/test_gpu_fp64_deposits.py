"""Deposits of the FP64 form behind optically thick cells: a beam through cells
whose optical depths run from 1e-3 to 45 with thin cells behind them, in a pure
absorber, every deposit against e^{-tau} (1 - e^{-dtau}).

The bound, relative for each cell, has no absolute part.  With faces right to half
an ulp and distances to an ulp, the length of a cell of 1/30 is off by 1e-14 of
itself; an optical depth of 170 in all is then off by 1.7e-12 at most, and by as
much again from its 60 additions: 3.4e-12 of e^{-tau}."""
import numpy as np
import pytest

from paper_1705_04702_gb300 import workloads as W

pytestmark = pytest.mark.gpu

THIN = [0.04, 0.3, 0.0624, 1e-3]
TAUS = {
    "thick_20": THIN + [20.0] + THIN * 3,
    "thick_30": THIN + [30.0] + THIN * 3,
    "thick_40": THIN + [40.0] + THIN * 3,
    "several": [3.0, 1e-3, 16.0, 1e-3, 5.0, 1e-3, 25.0, 1e-3, 37.0, 1e-3, 38.0, 1e-3, 45.0, 1e-3],
    "even": [0.49] * 60,
    "growing": list(np.geomspace(1e-3, 20.0, 60)),
}


@pytest.fixture(scope="module")
def S():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1705_04702_gb300 import build
    build.build()
    from paper_1705_04702_gb300 import skirt
    return skirt


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("name", sorted(TAUS))
def test_every_deposit_behind_thick_cells(S, name, axis):
    taus = np.array(TAUS[name])
    n = 60
    taus = np.concatenate([taus, np.full(n - taus.size, 0.01)])
    shape = [1, 1, 1]
    shape[axis] = n
    kr = (taus / (2.0 / n)).astype(np.float32)
    grid = W.Grid(*shape, (-1.0, 1.0, -1.0, 1.0, -1.0, 1.0), kr.reshape(shape[::-1]))
    pos, k = [0.1, -0.2, 0.3], [0.0, 0.0, 0.0]
    pos[axis], k[axis] = -1.0, 1.0
    prob = W.Problem("beam", grid, W.Source(W.SRC_BEAM, tuple(pos), tuple(k)), W.single_wavelength(albedo=0.0),
                     np.array([1], dtype=np.uint64), [], seed=3)
    got = S.run_problem(prob, precision=S.PREC_FP64)["absorbed"].cpu().numpy().ravel()
    d = kr.astype(np.longdouble) * (np.longdouble(2.0) / n)
    before = np.concatenate([[np.longdouble(0.0)], np.cumsum(d)[:-1]])
    want = (np.exp(-before) * -np.expm1(-d)).astype(np.float64)
    np.testing.assert_allclose(got, want, rtol=4e-12)
