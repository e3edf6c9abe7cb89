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


@pytest.mark.parametrize("variant", [oracle.FASGD, oracle.FASGD_STD])
@pytest.mark.parametrize("eps", [1e-4, 0.0])
@pytest.mark.parametrize("budget", [False, True])
def test_exact_mode_on_steps_far_below_theta(variant, eps, budget):
    """Gradients from subnormal up and quotients around 2^-66, where the pass
    relies on theta (2^-40 or more) not to change, with theta on both sides of
    that line, zero and subnormal: single pushes and a fused one, bit for bit."""
    torch, f = torch_cuda(), binding()
    rng = np.random.default_rng(66)
    P = 400_003
    line = np.float32(2.0 ** -40)
    edge = np.float32([line, np.nextafter(line, np.float32(0)), -line, 0.0, -0.0, 1e-45, -1e-40, 2.0 ** -66,
                       2.0 ** -41, 2.0 ** -39, 1.0, 2.0 ** 119, 2.0 ** 121])
    theta = np.where(rng.random(P) < 0.5, np.resize(edge, P), _wild(rng, P, -149, 10)).astype(np.float32)
    # Large n leaves v to its old value, so quotients spread over all exponents.
    n = np.where(rng.random(P) < 0.7, _wild(rng, P, 80, 99, False), _wild(rng, P, -30, 0, False)).astype(np.float32)
    b, v = np.zeros(P, np.float32), _wild(rng, P, -60, 60, False)
    grads = [_wild(rng, P, -149, -20), _wild(rng, P, -126, -60), _wild(rng, P, -149, 0), np.zeros(P, np.float32),
             _wild(rng, P, -100, -10)]
    grads[2][::3] = 0.0
    srv = f.Server(P, 4, 2.0 ** -3 * 1.1, variant, eps=eps)
    srv.set_exact(True)
    ora = oracle.OracleServer(P, 4, 2.0 ** -3 * 1.1, variant, eps=eps)
    srv.set_state(*[torch.from_numpy(x).cuda() for x in (theta, n, b, v)], 0)
    ora.theta[:], ora.n[:], ora.b[:], ora.v[:] = theta, n, b, v
    buf, dev = f.aligned_vectors(np.stack(grads))
    if budget:
        srv.set_tensors(streams.tensor_sizes(1, P, 5))
    with np.errstate(all="ignore"):
        for batch in ([0], [1], [2, 3, 4]):
            for k in batch:
                if budget and k < 2:
                    srv.push_budget(k % 4, 0, dev[k], P)
                else:
                    srv.push(k % 4, 0, dev[k])
                ora.push(k % 4, 0, grads[k])
            srv.apply_pending(len(batch))
            ora.apply_pending(len(batch))
            out = [torch.empty(P, device="cuda") for _ in range(4)]
            srv.get_state(*out)
            for name, x, y in zip(("theta", "n", "b", "v"), out, (ora.theta, ora.n, ora.b, ora.v)):
                _same_bits(x.cpu().numpy(), np.asarray(y, np.float32), (name, batch))
    srv.close()


def test_tiny_gradients_do_not_send_a_pass_the_long_way():
    """One gradient in a hundred 1e-22 times its size, as saturated outputs leave
    them: the exact pass takes about as long as without (it took 4.5 times as
    long while a lower bound on the gradient alone guarded it)."""
    torch, f = torch_cuda(), binding()
    P, K = 6_000_000, 8
    gen = torch.Generator("cuda").manual_seed(1)
    plain = [torch.randn(P, generator=gen, device="cuda") * 0.01 for _ in range(K)]
    tiny = [torch.where(torch.rand(P, generator=gen, device="cuda") < 0.01, g * 1e-22, g) for g in plain]
    start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = []
    for pool in (plain, tiny):
        srv = f.Server(P, 4, 1e-3, oracle.FASGD)
        srv.set_exact(True)
        srv.set_params(plain[0])
        times = []
        for _ in range(12):
            start.record()
            for k in range(K):
                srv.push(k % 4, srv.T, pool[k])
            srv.apply_pending(K)
            end.record()
            end.synchronize()
            times.append(start.elapsed_time(end))
        best.append(min(times))
        srv.close()
    assert best[1] < 2 * best[0], best
