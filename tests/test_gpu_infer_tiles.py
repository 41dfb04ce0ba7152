"""The surrogate's inference at the edges of its 32-row warp tiles and 16-row
halves: every row equals the row inferred alone bit for bit, whatever its tile
holds beside it, with live and empty rows mixed."""
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


@pytest.mark.parametrize("n", [1, 15, 16, 17, 31, 32, 33, 383, 384, 385, 60000])
def test_rows_do_not_depend_on_their_tile(S, n):
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    f = torch.randn((n, 32), device="cuda", generator=g) * 2.0 - 5.0
    tot = torch.rand(n, device="cuda", generator=g, dtype=torch.float64)
    tot[torch.rand(n, device="cuda", generator=g) < 0.3] = 0.0
    if n > 40:
        tot[16:32] = 0.0                          # an empty half
        tot[32:40] = 0.0
    net = S.MLP(seed=4)
    net.set_params(x_mean=np.full(32, -5.0, np.float32), x_std=np.full(32, 2.0, np.float32),
                   hull_lo=np.full(32, -9.0, np.float32), hull_hi=np.full(32, -1.0, np.float32))
    net.set_guard(0.9)
    em = torch.full((n, 100), float("nan"), dtype=torch.float64, device="cuda")
    fl = torch.full((n,), 7, dtype=torch.uint8, device="cuda")
    net.forward(f, tot, n, em, fl)
    out = ((f < -9.0) | (f > -1.0)).any(dim=1)
    e = 10.0 ** (f.double() - f.double().max(dim=1, keepdim=True).values)
    share = 1.0 / e.sum(dim=1)
    sure = (share - 0.9).abs() > 1e-5             # FP32 sums decide within a few ulp
    want = ((out | (share > 0.9)) & (tot > 0)).to(torch.uint8)
    assert torch.equal(fl[sure], want[sure])
    assert torch.all(em[tot == 0] == 0.0)
    np.testing.assert_allclose(em.sum(dim=1).cpu().numpy(), tot.cpu().numpy(), rtol=1e-5)
    pick = torch.unique(torch.cat([torch.arange(min(n, 40)), torch.arange(max(0, n - 5), n)])).tolist()
    for r in pick:
        one = torch.empty((1, 100), dtype=torch.float64, device="cuda")
        net.forward(f[r:r + 1].contiguous(), tot[r:r + 1].contiguous(), 1, one)
        assert torch.equal(one[0], em[r])
    net.close()
