"""Inference calls at once, each with its own network and stream, from several threads:
every call answers for itself (its rows, flags and status), as one at a time."""
import threading

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


def test_calls_of_several_networks_at_once(S):
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    sizes = (1, 31, 5000, 200_000)
    nets = [S.MLP(seed=k + 1) for k in range(len(sizes))]
    data, want = [], []
    for net, n in zip(nets, sizes):
        net.set_params(hull_lo=np.full(32, -2.0, np.float32), hull_hi=np.full(32, 2.0, np.float32))
        x = torch.randn((n, 32), device="cuda", generator=g)
        t = torch.rand(n, device="cuda", generator=g, dtype=torch.float64)
        em = torch.empty((n, 100), dtype=torch.float64, device="cuda")
        fl = torch.empty(n, dtype=torch.uint8, device="cuda")
        net.forward(x, t, n, em, fl)
        data.append((x, t, n))
        want.append((em, fl))
    got = [(torch.empty_like(e), torch.empty_like(f)) for e, f in want]
    streams = [torch.cuda.Stream() for _ in sizes]
    errors = []

    def call(k):
        try:
            for _ in range(20):
                nets[k].forward(*data[k], *got[k], stream=streams[k].cuda_stream)
        except Exception as e:  # reported below
            errors.append(e)

    torch.cuda.synchronize()
    threads = [threading.Thread(target=call, args=(k,)) for k in range(len(sizes))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for (e, f), (ge, gf) in zip(want, got):
        assert torch.equal(e, ge) and torch.equal(f, gf)
    for net in nets:
        net.close()


def test_an_empty_call_and_a_refused_one_leave_the_next_alone(S):
    import torch
    net = S.MLP(seed=1)
    x = torch.randn((40, 32), device="cuda")
    t = torch.ones(40, dtype=torch.float64, device="cuda")
    em = torch.empty((40, 100), dtype=torch.float64, device="cuda")
    net.forward(x, t, 0, em)
    odd = torch.empty(40 * 32 + 1, device="cuda")[1:]  # not on a 16-byte boundary: refused
    with pytest.raises(S.SkirtError):
        net.forward(odd, t, 40, em)
    net.forward(x, t, 40, em)
    np.testing.assert_allclose(em.sum(dim=1).cpu().numpy(), 1.0, rtol=1e-5)
    net.close()
