"""The mixed-form trace kernel's grid kinds and exits: an axis too long for
FP32 face indices against the ordinary Cartesian kernel, and traversals that
start in the last cell of an axis or tie at a grid edge against the oracle."""
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


def _long_problem(nx, npk=2000):
    """Unit cells, dust in the first 64 of nx along x, source among them."""
    kr = np.zeros((8, 8, nx), dtype=np.float32)
    kr[:, :, :64] = 0.2
    grid = W.Grid(nx, 8, 8, (0.0, float(nx), 0.0, 8.0, 0.0, 8.0), kr)
    return W.Problem("long", grid, W.Source(W.SRC_POINT, (20.3, 4.1, 3.7)), W.single_wavelength(),
                     np.array([npk], dtype=np.uint64), [W.Instrument(100.0, 60.0, 30.0, 100.0, 16)], seed=3)


def test_an_axis_of_2_23_cells_gives_the_short_axis_histories(S):
    """Beyond 2^23 cells per axis the kernel counts faces in integers.  Cells
    past the dust change no deposit, so the long grid's records are those of a
    4096-cell one bit for bit (the same planes, directions and densities)."""
    short = S.run_problem(_long_problem(4096), nrec=2000)
    full = S.run_problem(_long_problem((1 << 23) + 1), nrec=2000)
    a, b = short["records"].cpu().numpy(), full["records"].cpu().numpy()
    assert np.array_equal(a, b)
    nx = (1 << 23) + 1
    x = full["absorbed"].view(64, nx)[:, :64].cpu().numpy()
    y = short["absorbed"].view(64, 4096)[:, :64].cpu().numpy()
    np.testing.assert_allclose(x, y, rtol=1e-12)


@pytest.mark.parametrize("pos,direction", [
    ((0.9, 0.9, 0.9), (1.0, 0.0, 0.0)),              # one face from the grid's edge
    ((-0.9, 0.9, -0.9), (0.0, 0.0, -1.0)),
    ((0.0, 0.0, 0.0), (0.5773502691896258,) * 3),    # corner to corner: every crossing a three-way tie
    ((0.0, 0.0, 0.0), (0.7071067811865476, -0.7071067811865476, 0.0)),
])
@pytest.mark.parametrize("n", [1, 2, 7])
def test_beams_leave_the_grid_where_the_oracle_does(S, oracle_lib, pos, direction, n):
    """Deposits of a pure-absorber beam: the same cells, luminosities to the
    FP32 crossing lengths (1e-5 of the launch luminosity, the record bar)."""
    prob = W.beam_problem(W.uniform_grid(n, kr=0.7), pos, direction, npackets=3, albedo=0.0)
    ref = oracle_lib.trace(prob, nrec=3)
    g = S.run_problem(prob, nrec=3)
    np.testing.assert_allclose(g["absorbed"].cpu().numpy(), ref["absorbed"], rtol=0, atol=1e-5)
    np.testing.assert_allclose(g["records"].cpu().numpy()[..., :4], ref["records"][..., :4], rtol=0, atol=1e-5)
