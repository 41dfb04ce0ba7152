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


@pytest.mark.parametrize("nxyz,ext", [
    ((33, 5, 41), (4.0, 2.0, 0.5)),     # z cells the smallest: z runs fastest
    ((7, 40, 3), (2.0, 1.0, 3.0)),      # y cells
    ((1, 70, 9), (1.0, 1.0, 3.0)),      # y cells, one cell along x
    ((65, 3, 1), (6.5, 0.1, 3.0)),      # y cells, one cell along z
    ((64, 32, 33), (2.0, 2.0, 0.4)),
])
@pytest.mark.parametrize("nl", [1, 3, 4, 37])
def test_cell_orders_give_the_api_tables(S, nxyz, ext, nl):
    """Grids whose thinnest cells lie along y or z are traversed with that
    axis fastest.  The tables come back in the API's order: the FP64 form,
    which never reorders, gives them up to the <= 0.1% of packets whose FP32
    histories differ (each moves its luminosity once on either side: L1 2e-3),
    and an accumulating second call doubles them."""
    import torch
    nx, ny, nz = nxyz
    x = (np.arange(nx) + 0.5) / nx
    y = (np.arange(ny) + 0.5) / ny
    z = (np.arange(nz) + 0.5) / nz
    kr = (0.5 + 2.0 * x[None, None, :] + y[None, :, None] ** 2 + 0.3 * z[:, None, None]).astype(np.float32)
    ex, ey, ez = ext
    grid = W.Grid(nx, ny, nz, (0.0, ex, -ey, 0.0, 0.0, ez), kr)
    wl = W.single_wavelength() if nl == 1 else W.powerlaw_wavelengths(nl, 0.3, 3.0)
    prob = W.Problem("order", grid, W.Source(W.SRC_POINT, (0.31 * ex, -0.43 * ey, 0.57 * ez)), wl,
                     np.full(nl, 3000, dtype=np.uint64), [W.Instrument(100.0, 40.0, 20.0, 10.0, 8)], seed=11)
    a = S.run_problem(prob, precision=S.PREC_MIXED)
    b = S.run_problem(prob, precision=S.PREC_FP64)
    ta, tb = a["absorbed"].cpu().numpy(), b["absorbed"].cpu().numpy()
    assert np.abs(ta - tb).sum() <= 2e-3 * tb.sum()
    g = S.Grid(grid)
    outs = (torch.zeros_like(a["absorbed"]), torch.zeros_like(a["images_flat"]), torch.zeros_like(a["sed"]))
    S.run_problem(prob, grid=g, outputs=outs)
    S.run_problem(prob, grid=g, outputs=outs, accumulate=True, use_graph=True)
    np.testing.assert_allclose(outs[0].cpu().numpy(), 2.0 * ta, rtol=1e-12)
    g.close()


def _nested_tree(levels, p):
    """Leaves of every level: at each, the box that holds p (in [0, 1)^3) is split."""
    leaves, c = [], np.zeros(3, dtype=np.int64)
    for lev in range(1, levels + 1):
        kids = 2 * c + np.array([[o & 1, o >> 1 & 1, o >> 2 & 1] for o in range(8)])
        c = np.floor(np.array(p) * (1 << lev)).astype(np.int64)
        for k in kids:
            if lev == levels or (k != c).any():
                leaves.append([lev, *k])
    leaves = np.array(leaves, dtype=np.int32)
    kr = np.random.default_rng(levels).uniform(0.2, 1.0, len(leaves)).astype(np.float32)
    return W.Octree(levels, (-1.0, 1.0, -2.0, 2.0, 0.0, 1.0), leaves, kr)


@pytest.mark.parametrize("levels", [1, 2, 9, 15])
def test_nested_octrees_of_every_depth(S, levels):
    """Rays out of (and past) the finest leaf cross leaves of every level, up
    to the largest lattice the grid takes.  Pure-absorber beams deposit what
    the FP64 form does to the FP32 crossing lengths (1e-5 of the launch
    luminosity, the record bar); scattered packets up to the <= 0.1% whose FP32
    histories differ (L1 2e-3)."""
    p = (0.613, 0.427, 0.771)
    tree = _nested_tree(levels, p)
    src = (-1.0 + 2.0 * p[0], -2.0 + 4.0 * p[1], p[2])
    for d in [(1, 0, 0), (0, -1, 0), (0, 0, 1), (0.6, 0.8, 0), (-0.48, 0.64, -0.6), (0.36, -0.48, 0.8)]:
        prob = W.beam_problem(tree, src, d, npackets=2, albedo=0.0)
        a = S.run_problem(prob, precision=S.PREC_MIXED)["absorbed"].cpu().numpy()
        b = S.run_problem(prob, precision=S.PREC_FP64)["absorbed"].cpu().numpy()
        np.testing.assert_allclose(a, b, rtol=0, atol=1e-5)
    prob = W.Problem("nested", tree, W.Source(W.SRC_POINT, (src[0] + 0.3, src[1], src[2])), W.single_wavelength(),
                     np.array([4000], dtype=np.uint64), [W.Instrument(100.0, 40.0, 20.0, 5.0, 8)], seed=5)
    a = S.run_problem(prob, precision=S.PREC_MIXED)["absorbed"].cpu().numpy()
    b = S.run_problem(prob, precision=S.PREC_FP64)["absorbed"].cpu().numpy()
    assert np.abs(a - b).sum() <= 2e-3 * b.sum()
