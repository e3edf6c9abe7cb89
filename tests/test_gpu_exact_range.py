"""Exact arithmetic at the edges of the range in which the refined hardware
approximations are used: gradients, statistics and eps from subnormal to near
overflow, zeros of both signs, infinities and NaN, bit for bit against the
oracle (which computes every operation rounded once)."""

import numpy as np
import pytest

import oracle
from gpu_util import binding, torch_cuda
from paper_1601_04033_gb300 import streams

pytestmark = pytest.mark.gpu


def _wild(rng, P, lo, hi, signed=True):
    """Values with exponents spread over [lo, hi] and full mantissas."""
    x = np.ldexp(1.0 + rng.random(P), rng.integers(lo, hi + 1, P)).astype(np.float32)
    return x * rng.choice(np.float32([-1, 1]), P) if signed else x


def _same_bits(got, want, what):
    g, w = got.view(np.uint32), want.view(np.uint32)
    bad = np.nonzero((g != w) & ~(np.isnan(got) & np.isnan(want)))[0]
    assert bad.size == 0, (what, bad.size, bad[:4], got[bad[:4]], want[bad[:4]])


@pytest.mark.parametrize("variant", [oracle.FASGD, oracle.FASGD_STD])
@pytest.mark.parametrize("eps", [1e-4, 0.0, 2.0 ** -99, 2.0 ** -101, 1e-40, 2.0 ** 101])
@pytest.mark.parametrize("budget", [False, True])
def test_exact_mode_at_the_edges_of_its_fast_range(variant, eps, budget):
    torch, f = torch_cuda(), binding()
    rng = np.random.default_rng(17)
    P, edge = 40_003, np.float32([0.0, -0.0, 2.0 ** -60, 2.0 ** 60, 2.0 ** -61, 2.0 ** 61, 1e-45,
                                  -1e-45, 3e38, np.inf, -np.inf, np.nan, 2.0 ** -126, 1.0, -1.0])
    alpha = 2.0 ** -3
    theta = _wild(rng, P, -30, 10)
    theta[::7] = 0.0
    theta[1::7] = -0.0
    n, b = _wild(rng, P, -140, 100, False), _wild(rng, P, -80, 50)
    v = _wild(rng, P, -70, 70, False)
    grads = [_wild(rng, P, -140, 70), np.zeros(P, np.float32), np.resize(edge, P), -np.resize(edge[::-1], P)]
    srv = f.Server(P, 4, alpha, variant, eps=eps)
    srv.set_exact(True)
    ora = oracle.OracleServer(P, 4, alpha, variant, eps=eps)
    srv.set_state(*[torch.from_numpy(x).cuda() for x in (theta, n, b, v)], 0)
    ora.theta[:], ora.n[:], ora.b[:], ora.v[:] = theta, n, b, v
    buf, dev = f.aligned_vectors(np.stack(grads))
    if budget:       # a budget of P transmits every tensor: the ranged apply of the same rule
        srv.set_tensors(streams.tensor_sizes(1, P, 5))
    with np.errstate(all="ignore"):
        for k in range(4):
            if budget and k < 1:    # finite statistics: a budget push can be decided
                srv.set_hparams(0.95, 0.95, eps, 0.0, 1e-8, 0)
                srv.push_budget(k, 0, dev[k], P)
            else:
                srv.push(k, 0, dev[k])
            srv.apply_pending(1)
            ora.push(k, 0, grads[k])
            ora.apply_pending(1)
            out = [torch.empty(P, device="cuda") for _ in range(4)]
            srv.get_state(*out)
            for name, x, y in zip(("theta", "n", "b", "v"), out, (ora.theta, ora.n, ora.b, ora.v)):
                _same_bits(x.cpu().numpy(), np.asarray(y, np.float32), (name, k))
    srv.close()
