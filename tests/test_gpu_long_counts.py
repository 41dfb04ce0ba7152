"""Runs whose event cap allows a packet more crossings than a 32-bit counter holds
take a kernel that empties its counters at every event: the same histories, records
and counts as under the ordinary cap, on every grid kind."""
import dataclasses

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


@pytest.mark.parametrize("kind", ["torus", "octree", "long_axis"])
@pytest.mark.parametrize("precision", [0, 1])
def test_long_counts(S, kind, precision):
    if kind == "torus":
        prob = W.torus_problem(n=24, nlambda=3, packet_scale=5e-5, npx=16)
    elif kind == "octree":
        tree = W.refine_octree(W.disk_density(), (-24.0, 24.0, -24.0, 24.0, -24.0, 24.0), 5, 2, 2e-3)
        prob = W.octree_problem(tree, 2000, npx=16)
    else:  # an axis of more than 2^23 unit cells: face indices held as integers; dust in the first 64
        nx = (1 << 23) + 1
        kr = np.zeros((2, 2, nx), dtype=np.float32)
        kr[:, :, :64] = 0.4
        grid = W.Grid(nx, 2, 2, (0.0, float(nx), 0.0, 2.0, 0.0, 2.0), kr)
        prob = W.Problem("axis", grid, W.Source(W.SRC_POINT, (20.3, 1.1, 0.7)), W.single_wavelength(),
                         np.array([200], dtype=np.uint64), [W.Instrument(100.0, 60.0, 30.0, 100.0, 16)], seed=2)
    nrec = int(prob.npk.max())
    a = S.run_problem(prob, precision=precision, nrec=nrec)
    b = S.run_problem(dataclasses.replace(prob, max_events=2 ** 31 - 1), precision=precision, nrec=nrec)
    assert np.array_equal(a["records"].cpu().numpy(), b["records"].cpu().numpy())
    for k in ("scatterings", "deposit_steps", "locate_steps", "peel_steps"):
        assert a["ledger"][k] == b["ledger"][k]
