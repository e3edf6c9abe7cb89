"""The select kernels where their forms meet: around 850,000, 1.5M and 4.5M parameters
(more parameters per warp of the decision), around 8192 tiles of 4096
parameters (beyond, a scan kernel forms the tiles' places), at densities on
both sides of 256 kept entries per warp (fetched before or after the place is
known) and of 340 (a span that is read whole), every list bit for bit against
the oracle."""

import numpy as np
import pytest

import oracle
from gpu_util import binding, torch_cuda
from paper_1601_04033_gb300 import streams

pytestmark = pytest.mark.gpu
SWITCH = 8192 * 4096


# Kept entries per span of 1024, across every line in the compaction.
KEPT = [0, 1, 255, 256, 257, 339, 340, 341, 342, 511, 512, 1023, 1024, 341, 0, 1024, 339]


@pytest.mark.parametrize("P,c", [(SWITCH, 40.0), (SWITCH + 1, 40.0), (SWITCH - 4095, 40.0)]
                         + [(SWITCH, 0.0), (SWITCH + 1, 0.0), (SWITCH + 1, 12.0), (1_000_003, 12.0), (1_000_003, 0.0)]
                         + [(len(KEPT) * 1024 + tail, 1e4) for tail in (0, 3, 517, 1021)]
                         + [(P, 40.0) for P in (850_000, 850_001, 1_500_000, 1_500_001, 4_500_000, 4_500_001)]
                         + [(P, c) for P in (1, 31, 1023, 1025, 4095, 4097, 40_961)
                            for c in (0.0, 1.0, 30.0, 90.0, 1e4, float(2.0 ** 80), float("inf"))])
def test_select_lists_against_oracle(P, c):
    torch, f = torch_cuda(), binding()
    rng = np.random.default_rng(P % 9973)
    grad = rng.standard_normal(P, dtype=np.float32)
    v = np.exp(rng.random(P, dtype=np.float32) * np.float32(4.6))
    if P == 40_961:            # one warp all kept beside one with nothing kept
        v[1024:2048] = 1e30
        v[2048:3072] = 0.0
    if P // 1024 == len(KEPT):
        v[:] = 0.0             # kept with probability 1e-12, those below always
        for i, kept in enumerate(KEPT):
            v[1024 * i + rng.permutation(1024)[:kept]] = 1e30
        v[1024 * len(KEPT):] = 1e30
    srv = f.Server(P, 4, 0.001, f.FASGD, c_push=c, eps_b=1e-8, seed=11)
    g, vv = torch.from_numpy(grad).cuda(), torch.from_numpy(v).cuda()
    idx = torch.full((P,), -1, dtype=torch.int32, device="cuda")
    val = torch.zeros(P, device="cuda")
    cnt = torch.full((1,), -1, dtype=torch.int64, device="cuda")
    for n in range(2):         # twice: nothing carries over
        srv.select_compact(3, g, idx, val, cnt, v=vv)
        srv.sync()
        oi, ov = oracle.select(grad, v, c, 1e-8, 11, 3, n)
        m = int(cnt.item())
        assert m == oi.size
        assert np.array_equal(idx[:m].cpu().numpy(), oi)
        assert np.array_equal(val[:m].cpu().numpy().view(np.uint32), ov.view(np.uint32))
        assert (idx[m:] == -1).all() or n == 1
    srv.close()
