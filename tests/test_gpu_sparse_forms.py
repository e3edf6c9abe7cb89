"""The sparse apply on both sides of the switch between its forms (7M
parameters of host-side bound), at counts around its steps and around the
densities from which half and all of the large form's warps work, against the
oracle on the listed parameters; lists without a device count, short and empty."""

import numpy as np
import pytest

import oracle
from gpu_util import ATOL, RTOL, binding, torch_cuda

pytestmark = pytest.mark.gpu
SWITCH = 7_000_000
COUNTS = ((0, True), (1, False), (31, True), (33, False), (63, True), (257, True), (60_001, False),
          (700_003, True), (2_600_001, True))
# Large form: a sixteenth (SASGD), a seventh, nine twentieths of P, and all of it.
LINES = tuple((m, True) for m in (437_499, 437_500, 999_999, 1_000_000, 3_149_999, 3_150_000, SWITCH + 1))


@pytest.mark.parametrize("variant,exact", [(oracle.FASGD, False), (oracle.FASGD, True),
                                           (oracle.FASGD_STD, True), (oracle.SASGD, False)])
@pytest.mark.parametrize("P", [SWITCH, SWITCH + 1])
def test_both_forms(P, variant, exact):
    torch, f = torch_cuda(), binding()
    rng = np.random.default_rng(3)
    srv = f.Server(P, 4, 0.01, variant)
    srv.set_exact(exact)
    state = [rng.standard_normal(P, dtype=np.float32) * np.float32(0.01),
             rng.random(P, dtype=np.float32) * np.float32(1e-2), np.zeros(P, np.float32),
             rng.random(P, dtype=np.float32) * np.float32(50) + np.float32(1)]
    srv.set_state(*[torch.from_numpy(x).cuda() for x in state], 0)
    out = [torch.empty(P, device="cuda") for _ in range(4)]
    for m, device_count in COUNTS + (LINES if P > SWITCH else ()):
        keep = np.sort(rng.choice(P, m, replace=False)).astype(np.int32)
        g = (rng.standard_normal(m) * 0.05).astype(np.float32)
        idx = torch.zeros(P if device_count else max(m, 1), dtype=torch.int32, device="cuda")
        val = torch.zeros(idx.numel(), device="cuda")
        idx[:m], val[:m] = torch.from_numpy(keep).cuda(), torch.from_numpy(g).cuda()
        cnt = torch.tensor([m], dtype=torch.int64, device="cuda") if device_count else None
        srv.push_sparse(1, srv.T, idx, val, n_dev=cnt, n_max=P if device_count else m)
        srv.apply_pending(1)
        srv.sync()
        ora = oracle.OracleServer(max(m, 1), 4, 0.01, variant)
        ora.theta[:m], ora.n[:m], ora.b[:m], ora.v[:m] = (x[keep] for x in state)
        if m:
            ora.push(1, 0, g)
            ora.apply_pending(1)
            for x, y in zip(state, (ora.theta, ora.n, ora.b, ora.v)):
                x[keep] = y[:m]
        srv.get_state(*out)
        for k, (x, y) in enumerate(zip(out, state)):
            got = x.cpu().numpy()
            if exact or k in (1, 2):
                assert np.array_equal(got.view(np.uint32), y.view(np.uint32)), (m, k)
            else:
                assert (np.abs(got - y) <= RTOL * np.abs(y) + ATOL).all(), (m, k)
        state = [x.cpu().numpy() for x in out]
    srv.close()
