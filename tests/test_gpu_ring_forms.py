"""Every form of the dense pass by K (slices per stage, stages, consumers, plain
grid): one fused pass of K pushes equals K passes of one push bit for bit, for
each rule and arithmetic, with ragged sizes on both sides of the plain grid's
limit and beyond L2 (the passes of one push are compared with the oracle elsewhere)."""

import pytest

from gpu_util import binding, ring_P, torch_cuda

pytestmark = pytest.mark.gpu
FORMS = [("sasgd", 1, False), ("fasgd", 2, False), ("fasgd exact", 2, True),
         ("std", 3, False), ("std exact", 3, True)]


@pytest.mark.parametrize("name,variant,exact", FORMS)
@pytest.mark.parametrize("where", ["grid", "ring in L2", "ring from HBM"])
def test_fused_pass_equals_single_pushes(name, variant, exact, where):
    torch, f = torch_cuda(), binding()
    P = {"grid": 300_003, "ring in L2": ring_P(70_001), "ring from HBM": 16_300_003}[where]
    gen = torch.Generator(device="cuda").manual_seed(variant + 10 * exact)
    buf = torch.zeros((33, (P + 3) // 4 * 4), device="cuda")
    rows = [buf[k, :P] for k in range(33)]
    for x in rows:
        x.normal_(generator=gen).mul_(0.03)
    rows[32].mul_(0.5)
    a, b = (f.Server(P, 4, 1e-3, variant) for _ in range(2))
    out = [[torch.empty(P, device="cuda") for _ in range(4)] for _ in range(2)]
    for s in (a, b):
        s.set_exact(exact)
        s.set_params(rows[32])
    T = 0
    for K in [*range(1, 18), 24, 31, 32]:
        js = [max(0, T - (5 * k) % 7) for k in range(K)]
        for k in range(K):
            a.push(k % 4, js[k], rows[(k + K) % 32])
        a.apply_pending(K)
        for k in range(K):
            b.push(k % 4, js[k], rows[(k + K) % 32])
        for _ in range(K):
            b.apply_pending(1)
        T += K
        a.get_state(*out[0])
        b.get_state(*out[1])
        for x, y, what in zip(*out, ("theta", "n", "b", "v")):
            assert torch.equal(x.view(torch.int32), y.view(torch.int32)), (name, K, what)
    a.sync()
    b.sync()
    a.close()
    b.close()
