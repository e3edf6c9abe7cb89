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


def test_copies_past_an_allocation_are_refused():
    """A device range that runs past its allocation is refused on the host, as
    the runtime's copies refuse it, and leaves the server usable; a range up to
    an allocation's last byte is written.  Checked only where the driver says
    that nothing is mapped behind the buffer."""
    import ctypes
    import torch
    from paper_1601_04033_gb300 import fasgd
    P, size = 70_003, 64 << 20
    cuda = ctypes.CDLL("libcuda.so.1")
    torch.cuda.synchronize()
    srv = fasgd.Server(P, 2, 0.01, fasgd.FASGD)
    want = np.random.default_rng(1).standard_normal(P).astype(np.float32)
    srv.set_state(*[torch.from_numpy(want)] * 4, 3)
    base, got, n = ctypes.c_uint64(), ctypes.c_uint64(), ctypes.c_size_t()
    assert cuda.cuMemAlloc_v2(ctypes.byref(base), ctypes.c_size_t(size)) == 0
    try:
        end = base.value + size
        assert cuda.cuMemGetAddressRange_v2(ctypes.byref(got), ctypes.byref(n), ctypes.c_uint64(base.value)) == 0
        assert (got.value, n.value) == (base.value, size)
        fits = end - 4 * P
        assert fasgd.fasgd_pull(srv.h, fits)[0] == fasgd.OK
        assert fasgd.fasgd_get_state(srv.h, None, fits, None, None)[0] == fasgd.OK
        host = np.empty(P, np.float32)
        assert cuda.cuMemcpyDtoH_v2(host.ctypes.data_as(ctypes.c_void_p), ctypes.c_uint64(fits), ctypes.c_size_t(4 * P)) == 0
        assert np.array_equal(host, want)
        if cuda.cuMemGetAddressRange_v2(ctypes.byref(got), ctypes.byref(n), ctypes.c_uint64(end)) != 0:
            for p in (fits + 4, end - 4, end - 4 * (P // 2)):
                assert fasgd.fasgd_pull(srv.h, p)[0] == fasgd.ECUDA
                assert fasgd.fasgd_get_state(srv.h, p, None, None, None)[0] == fasgd.ECUDA
                assert fasgd.fasgd_get_state(srv.h, None, fits, None, p)[0] == fasgd.ECUDA
    finally:
        assert cuda.cuMemFree_v2(base) == 0
    out = torch.zeros(P, device="cuda")
    assert srv.pull(out) == 3
    srv.sync()
    assert np.array_equal(out.cpu().numpy(), want)
    srv.close()


def test_pull_under_capture():
    import torch
    from paper_1601_04033_gb300 import fasgd
    P = 10_007
    srv = fasgd.Server(P, 2, 0.01, fasgd.FASGD)
    out = torch.zeros(P, device="cuda")
    s = torch.cuda.Stream()
    srv.set_stream(s)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(s):
        srv.pull(out)
    s.synchronize()
    with torch.cuda.graph(graph, stream=s):
        srv.pull(out)
    want = torch.arange(P, dtype=torch.float32)
    srv.set_params(want)
    s.synchronize()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out.cpu(), want)
    srv.close()
