"""fasgd_pull and fasgd_get_state into device buffers: the copy kernel's sizes
(remainders of quads and blocks, both unrolls) and destination alignments,
against the values that were set, and host and device destinations mixed."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [1, 3, 4, 5, 1023, 1025, 4096, 4099, 152 * 8 * 256 * 4 + 3, 2_500_001]


@pytest.mark.parametrize("shift", [0, 1, 2])
@pytest.mark.parametrize("P", SIZES)
def test_pull_and_state_copies(P, shift):
    import torch
    from paper_1601_04033_gb300 import fasgd
    rng = np.random.default_rng(P + shift)
    want = [rng.standard_normal(P).astype(np.float32) for _ in range(4)]
    srv = fasgd.Server(P, 2, 0.01, fasgd.FASGD)
    srv.set_state(*[torch.from_numpy(w) for w in want], 5)
    guard = [torch.full((P + 8,), 7.0, device="cuda") for _ in range(4)]
    out = [x[shift:shift + P] for x in guard]
    assert srv.pull(out[0]) == 5
    assert np.array_equal(out[0].cpu().numpy(), want[0])
    assert srv.get_state(*out) == 5
    for x, full, w in zip(out, guard, want):
        assert np.array_equal(x.cpu().numpy(), w)
        assert (full[:shift] == 7).all() and (full[shift + P:] == 7).all()
    host = [torch.zeros(P), None, torch.zeros(P, device="cuda"), torch.zeros(P)]
    srv.get_state(*host)
    for x, w in zip(host, want):
        assert x is None or np.array_equal(x.cpu().numpy(), w)
    pinned = torch.zeros(P, pin_memory=True)
    srv.pull(pinned)
    srv.sync()
    assert np.array_equal(pinned.numpy(), want[0])
    srv.close()
