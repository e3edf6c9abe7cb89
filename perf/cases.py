"""What is measured: the work a user of the parameter server has it do.

Every case is one turn of the server's protocol through the public binding
(`paper_1601_04033_gb300.fasgd.Server`, `fasgd.fetch_apply`, `sim.Simulation`),
in one of five kinds:

* ``dense``     K clients push whole gradients, the server applies them in one
                call and hands the parameters back (`push` x K, `apply_pending(K)`,
                `pull`).  ``source="host"``: gradients and the pulled parameters
                live in pinned host memory (`push_host`).  ``exact``: correctly
                rounded arithmetic.  ``checkpoint``: the server's whole state is
                also read back (`get_state`), as when a run is saved.
* ``exchange``  B-FASGD per parameter, four clients in turn: each selects and
                compacts what it sends, the server applies the list, the client
                selects what it fetches and scatters it into its copy; then the
                server's parameters are pulled for evaluation.
* ``message``   B-FASGD with one decision per message: a round of eight clients
                push, the server applies, the eight fetch; then a pull.
* ``budget``    B-FASGD per tensor under a bandwidth budget: four clients' pushes
                and fetches in turn, then a pull.
* ``sim``       the closed-loop simulation: a run of eight dispatcher batches
                (gradient at the client's copy, server pass, refresh) and the
                loss at its end.

Sizes are those of the package's own workloads (7,850: softmax regression;
159,010: the 784-200-10 network; 1,290,510: 784-1000-500-10; 25 million; 2^28)
and odd ones between them.  Servers start from a state in the middle of
training: n, b, v as running averages of the gradients that follow.
"""

from __future__ import annotations

import math

import numpy as np
import torch

GAMMA, BETA, EPS, EPS_B = 0.95, 0.95, 1e-4, 1e-8
RULES = {"asgd": 0, "sasgd": 1, "fasgd": 2, "fasgd-std": 3}
# Learning rates: the best ones the paper reports for FASGD and SASGD (Sec. 4.1),
# and the simulation's (its quadratic has curvatures up to 10).
ALPHA = {"asgd": 0.01, "sasgd": 0.04, "fasgd": 0.005, "fasgd-std": 0.005}
SIM_ALPHA = {"asgd": 0.01, "sasgd": 0.03, "fasgd": 0.03, "fasgd-std": 0.001}
T0 = 1000                      # the server's timestamp when a case starts
SEND, FETCH = 0.2, 0.1         # 5x fewer pushed entries, 10x fewer fetched ones
ROUND = {"exchange": 4, "message": 8, "budget": 4}      # clients in a turn
SIM_BATCHES = 8


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _dense(P, K, rule="fasgd", exact=False, source="device", checkpoint=False, lam=128):
    return {"kind": "dense", "P": P, "K": K, "rule": rule, "exact": exact, "source": source,
            "checkpoint": checkpoint, "lam": lam}


def _exchange(P, rule="fasgd", lam=64, live=True):
    return {"kind": "exchange", "P": P, "rule": rule, "lam": lam, "live": live}


def _message(P, rule="fasgd", lam=64):
    return {"kind": "message", "P": P, "rule": rule, "lam": lam}


def _budget(P, tensors, rule="fasgd", lam=64):
    return {"kind": "budget", "P": P, "rule": rule, "lam": lam, "tensors": tensors}


def _sim(P, lam, K, rule="fasgd", fetch="full", tensors=0):
    return {"kind": "sim", "P": P, "rule": rule, "lam": lam, "K": K, "fetch": fetch,
            "tensors": tensors}


def listed():
    return [
        # The smallest model, one push at a time: what a call costs.
        {"name": "dense-7850-k1", **_dense(7_850, 1, lam=4)},
        # A mid-sized network, one push at a time: the state stays in L2.
        {"name": "dense-1.29m-k1", **_dense(1_290_510, 1, lam=32)},
        # An odd size past the on-chip caches, five pushes, the whole state saved.
        {"name": "dense-5m-std-k5-save", **_dense(5_000_003, 5, rule="fasgd-std", checkpoint=True)},
        # The main workload.
        {"name": "dense-25m-k8", **_dense(25_000_000, 8)},
        # The same where runs must reproduce bit for bit on any IEEE machine.
        {"name": "dense-25m-k8-exact", **_dense(25_000_000, 8, exact=True)},
        # The largest model.
        {"name": "dense-268m-k16", **_dense(268_435_456, 16, lam=256)},
        # Clients on the other side of the host link.
        {"name": "dense-5m-sasgd-k4-host", **_dense(5_000_011, 4, rule="sasgd", source="host")},
        # Bandwidth-reduced exchanges of a large and of a mid-sized model.
        {"name": "exchange-25m", **_exchange(25_000_000)},
        {"name": "exchange-1.29m", **_exchange(1_290_510, live=False)},
        {"name": "message-25m", **_message(25_000_000)},
        {"name": "budget-25m", **_budget(25_000_000, 160)},
        # The paper's own experiment loop, at its network's size.
        {"name": "sim-159k", **_sim(159_010, 32, 1)},
    ]


def _log_size(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng):
    rule = rng.choice(["fasgd", "fasgd", "fasgd", "sasgd", "asgd", "fasgd-std"])
    lam = rng.choice([4, 16, 32, 64])
    kind = rng.choice(["dense"] * 7 + ["exchange"] * 4 + ["message"] * 3 + ["budget"] * 3 + ["sim"] * 3)
    if kind == "dense":
        K = rng.choice([1, 1, 2, 3, 4, 5, 8, 8, 13, 16, 32])
        how = rng.random()
        if how < 0.15:
            return _dense(_log_size(rng, 1_000, 8_000_000), min(K, 8), rule, source="host", lam=lam)
        exact = how < 0.35
        return _dense(_log_size(rng, 1_000, 64_000_000), K, rule, exact=exact,
                      checkpoint=rng.random() < 0.15, lam=lam)
    if kind == "exchange":
        return _exchange(_log_size(rng, 5_000, 40_000_000), rule, lam, rng.random() < 0.5)
    if kind == "message":
        return _message(_log_size(rng, 5_000, 30_000_000), rule, lam)
    if kind == "budget":
        T = rng.choice([2, 8, 17, 64, 160, 400])
        return _budget(_log_size(rng, 10_000, 40_000_000), T, rule, lam)
    P = _log_size(rng, 5_000, 1_000_000)
    fetch = rng.choice(["full", "full", "param", "message", "budget"])
    return _sim(P, max(4, min(lam, 16_000_000 // P)), rng.choice([1, 1, 2, 4]), rule, fetch,
                16 if fetch == "budget" else 0)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _rand(seed, tag, device="cuda"):
    g = torch.Generator(device=device)
    g.manual_seed((seed * 1_000_003 + tag) & 0x7FFF_FFFF_FFFF)
    return g


def _rows(R, P):
    """R fp32 vectors of length P, each starting on a 16-byte boundary."""
    buf = torch.zeros((R, (P + 3) // 4 * 4), dtype=torch.float32, device="cuda")
    return [buf[r, :P] for r in range(R)]


def _sizes(P, T, seed):
    """T tensors with the size mix of a layered network: weights over three
    decades, vectors of 16 to 4096."""
    g = np.random.default_rng((seed, 77))
    vec = np.exp(g.uniform(math.log(16), math.log(4096), T // 2))
    vec = np.maximum(1, np.floor(vec * min(1.0, (P / 4) / max(1.0, vec.sum())))).astype(np.int64)
    w = np.exp(g.uniform(0.0, math.log(1000.0), T - T // 2))
    rest = P - int(vec.sum())
    mat = np.maximum(1, np.floor(w / w.sum() * (rest - w.size))).astype(np.int64)
    mat[int(np.argmax(mat))] += rest - int(mat.sum())
    out = np.empty(T, np.int64)
    out[0::2], out[1::2] = mat, vec
    return out


def _slots(case):
    """Gradients kept: two turns' worth while that is small."""
    K = case["K"] if case["kind"] == "dense" else ROUND[case["kind"]]
    return K if 8 * K * case["P"] > (4 << 30) else 2 * K


def _delays(case, seed):
    """Step-staleness of the pushes: failures before the first success, p = 0.05."""
    return (np.random.default_rng((seed, 5)).geometric(0.05, 64) - 1).tolist()


def _mid_training(case, seed):
    """theta, n, b, v in the middle of a run, and the gradients to come:
    g = m + s z, m ~ N(0, 1e-3^2), s log-uniform in [1e-4, 1e-1] (per tensor
    also scaled by up to 10 either way, as layers differ)."""
    P, R, g = case["P"], _slots(case), _rand(seed, 1)
    std_rule = case["rule"] == "fasgd-std"
    m = torch.randn(P, generator=g, device="cuda").mul_(1e-3)
    s = torch.rand(P, generator=g, device="cuda").mul_(math.log(1e3)).add_(math.log(1e-4)).exp_()
    if case.get("tensors"):
        f = np.exp(np.random.default_rng((seed, 6)).uniform(-math.log(10), math.log(10), case["tensors"]))
        s.mul_(torch.repeat_interleave(torch.tensor(f, dtype=torch.float32, device="cuda"),
                                       torch.tensor(_sizes(P, case["tensors"], seed), device="cuda")))
    th, n, b, v = _rows(4, P)
    th.normal_(generator=g).mul_(0.01)
    b.normal_(generator=g).mul_(0.16).mul_(s).add_(m)          # mean over ~ 1 / (1 - gamma) pushes
    torch.mul(b, b, out=n)
    n.addcmul_(s, s)
    torch.addcmul(n, b, b, value=-1, out=v)
    v.clamp_(min=0).add_(EPS).sqrt_()
    if not std_rule:
        v.reciprocal_()
    grads = _rows(R, P)
    for x in grads:
        x.normal_(generator=g).mul_(s).add_(m)
    return th, n, b, v, grads


def _threshold(v, share):
    """c of Eq. 9 at which the expected share mean v / (v + c) is sent."""
    a = v[:: max(1, v.numel() // 65_536)].double().cpu().numpy() + EPS_B
    lo, hi = 0.0, float(a.max()) / share
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if float(np.mean(a / (a + mid))) > share else (lo, mid)
    return float(np.float32(0.5 * (lo + hi)))


def _mean_threshold(v, share):
    return float(np.float32(float(v.double().mean()) * (1.0 / share - 1.0)))


def _copies(case, seed, th):
    """The clients' own, slightly older parameters."""
    g, out = _rand(seed, 2), _rows(ROUND[case["kind"]], case["P"])
    for x in out:
        x.normal_(generator=g).mul_(1e-3).add_(th)
    return out


def _client_v(v, seed):
    """A client's own, slightly older copy of v."""
    out = _rows(1, v.numel())[0]
    out.normal_(generator=_rand(seed, 3)).mul_(0.05).exp_().mul_(v)
    return out


def _objective(case, seed):
    """The simulation's quadratic (curvature, minimiser, noise; numpy)."""
    P, g = case["P"], np.random.default_rng((seed, 9))
    h = np.exp(g.uniform(math.log(1e-2), math.log(10.0), P)).astype(np.float32)
    star = (g.standard_normal(P, dtype=np.float32) * np.float32(0.1))
    sigma = np.exp(g.uniform(math.log(1e-3), math.log(1e-1), P)).astype(np.float32)
    th = g.standard_normal(P, dtype=np.float32) * np.float32(0.01)
    sched = np.stack([g.permutation(case["lam"])[: case["K"]] for _ in range(64 * SIM_BATCHES)])
    return h, star, sigma, th, sched.astype(np.int32)


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------
def prepare(case, seed):
    from paper_1601_04033_gb300 import fasgd, sim
    P, kind, rule = case["P"], case["kind"], RULES[case["rule"]]
    st = {"case": case, "turn": 0, "push": 0}
    if kind == "sim":
        h, star, sigma, th, sched = _objective(case, seed)
        sizes = _sizes(P, case["tensors"], seed) if case["tensors"] else None
        st["sim"] = sim.Simulation(P, case["lam"], SIM_ALPHA[case["rule"]], rule, K=case["K"],
                                   seed=seed, fetch=case["fetch"], objective=(h, star, sigma),
                                   theta0=th, c_fetch=1.0 if case["fetch"] in ("param", "message") else 0.0,
                                   tensor_sizes=sizes, fetch_budget=P // 4 if sizes is not None else None)
        st["sched"] = sched
        return st
    th, n, b, v, grads = _mid_training(case, seed)
    srv = fasgd.Server(P, case["lam"], ALPHA[case["rule"]], rule, seed=seed)
    srv.set_state(th, n, b, v, T0)
    st.update(srv=srv, T=T0, d=_delays(case, seed), grads=grads)
    if kind == "dense":
        srv.set_exact(case["exact"])
        if case["source"] == "host":
            st["grads"] = [x.cpu().pin_memory() for x in grads]
            st["out"] = torch.empty(P, pin_memory=True)
        else:
            st["out"] = torch.empty(P, device="cuda")
        if case["checkpoint"]:
            st["save"] = [torch.empty(P, device="cuda") for _ in range(4)]
        return st
    st["copies"] = _copies(case, seed, th)
    st["out"] = torch.empty(P, device="cuda")
    if kind == "exchange":
        srv.set_hparams(GAMMA, BETA, EPS, _threshold(v, SEND), EPS_B, seed)
        srv.set_fetch_threshold(_threshold(v, FETCH))
        st["v"] = None if case["live"] else _client_v(v, seed)
        for k in ("push", "fetch"):
            st[k + "_list"] = (torch.zeros(P, dtype=torch.int32, device="cuda"),
                               torch.zeros(P, device="cuda"),
                               torch.zeros(1, dtype=torch.int64, device="cuda"))
    elif kind == "message":
        srv.set_hparams(GAMMA, BETA, EPS, _mean_threshold(v, SEND), EPS_B, seed)
        srv.set_fetch_threshold(_mean_threshold(v, FETCH))
        for k in ("sent", "fetched"):
            st[k] = torch.zeros(ROUND[kind], dtype=torch.int32, device="cuda")
            st[k + "_at"] = list(st[k].split(1))
    else:
        sizes = _sizes(P, case["tensors"], seed)
        srv.set_tensors(sizes)
        for k in ("push", "fetch"):
            st[k + "_out"] = (torch.zeros(case["tensors"], dtype=torch.uint8, device="cuda"),
                              torch.zeros(1, device="cuda"),
                              torch.zeros(1, dtype=torch.int64, device="cuda"))
    return st


def _next(st):
    """Client, timestamp and gradient of the next push."""
    t, case = st["push"], st["case"]
    st["push"] = t + 1
    return t % case["lam"], max(0, st["T"] - st["d"][t % 64]), st["grads"][t % len(st["grads"])]


def run(st):
    case = st["case"]
    kind, P = case["kind"], case["P"]
    turn = st["turn"]
    st["turn"] = turn + 1
    if kind == "sim":
        at = turn % 64 * SIM_BATCHES
        losses = st["sim"].run(st["sched"][at:at + SIM_BATCHES])
        return {"loss": losses, "clients": list(st["sim"].clients[:8])}
    srv = st["srv"]
    if kind == "dense":
        push = srv.push_host if case["source"] == "host" else srv.push
        for _ in range(case["K"]):
            push(*_next(st))
        srv.apply_pending(case["K"])
        st["T"] = srv.pull(st["out"])
        if case["checkpoint"]:
            srv.get_state(*st["save"])
            return {"theta": st["out"], "state": st["save"]}
        return {"theta": st["out"]}
    copies, who = st["copies"], [_next(st) for _ in range(ROUND[kind])]
    if kind == "exchange":
        from paper_1601_04033_gb300 import fasgd
        (pi, px, pn), (fi, fx, fn) = st["push_list"], st["fetch_list"]
        for (c, j, grad), mine in zip(who, copies):
            srv.select_compact(c, grad, pi, px, pn, v=st["v"])
            srv.push_sparse(c, j, pi, px, n_dev=pn, n_max=P)
            srv.apply_pending(1)
            srv.fetch_compact(c, fi, fx, fn, v=st["v"])
            fasgd.fetch_apply(mine, fi, fx, n_dev=fn, n_max=P)
        out = {"push": st["push_list"], "fetch": st["fetch_list"]}
    elif kind == "message":
        for (c, j, grad), sent in zip(who, st["sent_at"]):
            srv.push_message(c, j, grad, sent)
        srv.apply_pending(len(who))
        for (c, _, _), mine, fetched in zip(who, copies, st["fetched_at"]):
            srv.fetch_message(c, mine, fetched)
        out = {"sent": st["sent"], "fetched": st["fetched"]}
    else:
        for (c, j, grad), mine in zip(who, copies):
            srv.push_budget(c, j, grad, int(SEND * P), *st["push_out"])
            srv.apply_pending(1)
            srv.fetch_budget(c, mine, int(FETCH * P), *st["fetch_out"])
        out = {"push": st["push_out"], "fetch": st["fetch_out"]}
    st["T"] = srv.pull(st["out"])
    out.update(copies=copies, theta=st["out"])
    return out


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    P, kind = case["P"], case["kind"]
    fas = case["rule"] in ("fasgd", "fasgd-std")
    state = 32 if fas else 8                    # theta (n, b, v) read and written
    flops = 19 if fas else 2                    # a push's arithmetic on one parameter
    if kind == "dense":
        K = case["K"]
        save = (16 if fas else 4) if case["checkpoint"] else 0
        return {"bytes": P * (state + 4 * K + 4 + save), "flops": P * K * flops}
    turns = ROUND.get(kind)
    if kind == "exchange":
        # The statistic once for each decision, the gradient's and theta's kept
        # entries, both lists, the state where an entry was sent, the client's copy.
        one = 8 + SEND * (4 + 8 + state) + FETCH * (4 + 8 + 4)
        return {"bytes": P * (turns * one + 8), "flops": P * turns * (SEND * flops + 2 * 12)}
    if kind == "message":
        # The pass with its gradient, a sent gradient's slot, a fetched copy.
        one = state + 4 + SEND * 4 + FETCH * 8
        return {"bytes": P * (turns * one + 4), "flops": P * turns * flops}
    if kind == "budget":
        one = SEND * (state + 4) + FETCH * 8
        return {"bytes": P * (turns * one + 8), "flops": P * turns * SEND * flops}
    K = case["K"]
    fetch = {"full": 8, "param": 16, "message": 8, "budget": 2}[case["fetch"]]
    batch = K * (20 + fetch) + state + 4 * K
    return {"bytes": SIM_BATCHES * P * batch + 12 * P, "flops": SIM_BATCHES * P * K * (flops + 8)}


def tolerance(case):
    # Measured against exact(): 0.2e-7 to 1.0e-7 on every kind (32-bit sums of
    # steps small beside theta), up to 1.1e-7 on the simulation's clients.
    # Decisions, lists and counts are whole numbers: the same.
    return {"rel": 2e-6 if case["kind"] == "sim" else 5e-7}


# ---------------------------------------------------------------------------
# the same in 64 bits, without the package
# ---------------------------------------------------------------------------
def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon et al., SC'11) on int64 tensors holding 32-bit words."""
    k0, k1, m = seed & 0xFFFFFFFF, seed >> 32 & 0xFFFFFFFF, 0xFFFFFFFF

    def mul(a, x):
        t = a * (x & 0xFFFF)
        w = a * (x >> 16) + (t >> 16)
        return w >> 16, (w & 0xFFFF) << 16 | t & 0xFFFF

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c0)
        h1, l1 = mul(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = k0 + 0x9E3779B9 & m, k1 + 0xBB67AE85 & m
    return c0, c1, c2, c3


def _words(P, client, n, seed):
    """The draw word of each parameter."""
    q = torch.arange((P + 3) // 4, dtype=torch.int64, device="cuda")
    z = torch.zeros_like(q)
    return torch.stack(_philox(q, z + client, z + (n & 0xFFFFFFFF), z + (n >> 32), seed), 1).reshape(-1)[:P]


def _one_word(counter, client, n, seed):
    t = [torch.tensor([x], dtype=torch.int64) for x in (counter, client, n & 0xFFFFFFFF, n >> 32)]
    return [int(w) for w in _philox(*t, seed)]


def _passes(word, v, c):
    """Eq. 9, exactly: u / 2^24 < 1 / (1 + c / a), a and a + c rounded to 32 bits."""
    a = v.float() + torch.tensor(EPS_B, dtype=torch.float32, device=v.device)
    d = a + torch.tensor(c, dtype=torch.float32, device=v.device)
    return (word >> 8).double() * d.double() < a.double() * 16777216.0


def _apply(rule, alpha, x, g, tau):
    """One push on 64-bit theta, n, b, v (in place).  The hyper-parameters are
    the 32-bit numbers the server was given."""
    f = np.float32
    if rule == "asgd":
        x[0].sub_(g * float(f(alpha)))
        return
    coef = float(f(alpha)) / max(tau, 1)
    if rule == "sasgd":
        x[0].sub_(g * coef)
        return
    th, n, b, v = x
    ga, be = float(f(GAMMA)), float(f(BETA))
    n.mul_(ga).addcmul_(g, g, value=1 - ga)
    b.mul_(ga).add_(g, alpha=1 - ga)
    r = (n - b * b).clamp_(min=0).add_(float(f(EPS))).sqrt_()
    if rule == "fasgd":
        r.reciprocal_()
    v.mul_(be).add_(r, alpha=1 - be)
    th.addcdiv_(g, v, value=-coef)


def _smallest_c(sizes, vbar, budget, P):
    """The smallest 32-bit c with sum_t floor(s_t a_t / (a_t + c) 2^32) <= budget 2^32."""
    s, a = [int(x) for x in sizes], np.asarray(vbar, np.float32) + np.float32(EPS_B)

    def spent(x):
        q = a / (a + x)
        return sum((k * int(np.float64(y) * 2.0 ** 60)) >> 28 for k, y in zip(s, q))

    lo, hi = -1, 0x7F800000
    while hi - lo > 1:
        mid = (lo + hi) // 2
        x = np.array(mid, np.uint32).view(np.float32)
        lo, hi = (lo, mid) if spent(x) <= min(budget, P) << 32 else (mid, hi)
    return float(np.array(hi, np.uint32).view(np.float32))


def _exact_sim(case, seed):
    if case["fetch"] != "full":       # decisions on rounded statistics: no 64-bit value
        return None
    P, K = case["P"], case["K"]
    h, star, sigma, th, sched = _objective(case, seed)
    h, star, sigma, th = (torch.tensor(x, dtype=torch.float64, device="cuda") for x in (h, star, sigma, th))
    x = [th] + [torch.zeros_like(th) for _ in range(3)]
    copies, at, count, T = [th.clone() for _ in range(case["lam"])], [0] * case["lam"], [0] * case["lam"], 0
    root12 = float(np.float32(math.sqrt(12.0)))
    for batch in sched[:SIM_BATCHES]:
        todo = []
        for c in batch.tolist():
            w = _words(P, c + (1 << 30), count[c], seed)
            xi = (((w >> 9).double() + 0.5) / 8388608.0 - 0.5) * root12
            todo.append((h * (copies[c] - star) + sigma * xi, at[c]))
            count[c] += 1
        for k, (g, j) in enumerate(todo):
            _apply(case["rule"], SIM_ALPHA[case["rule"]], x, g, T + k - j)
        T += K
        for c in batch.tolist():
            copies[c].copy_(x[0])
            at[c] = T
    loss = 0.5 * (h * (x[0] - star) ** 2).sum()
    return {"loss": loss.reshape(1), "clients": copies[:8]}


def exact(case, seed):
    P, kind, rule = case["P"], case["kind"], case["rule"]
    if kind == "sim":
        return _exact_sim(case, seed)
    th, n, b, v, grads = _mid_training(case, seed)
    d, alpha, lam = _delays(case, seed), ALPHA[rule], case["lam"]
    # Push t of the first turn is applied at T0 + t; its timestamp counts from T0
    # (a B-FASGD client of an exchange is told the same).
    tau = [min(d[t % 64], T0) + t for t in range(64)]
    if kind == "dense":
        out = [torch.empty(P, dtype=torch.float64, device="cuda") for _ in range(4 if case["checkpoint"] else 1)]
        for lo in range(0, P, 1 << 24):
            part = slice(lo, min(P, lo + (1 << 24)))
            x = [y[part].double() for y in (th, n, b, v)]
            for k in range(case["K"]):
                _apply(rule, alpha, x, grads[k][part].double(), tau[k])
            for y, z in zip(out, x):
                y[part] = z
        if case["checkpoint"]:
            return {"theta": out[0], "state": out}
        return {"theta": out[0]}
    x = [y.double() for y in (th, n, b, v)]
    copies = _copies(case, seed, th)
    if kind == "exchange":
        mine = v if case["live"] else _client_v(v, seed)
        cp, cf = _threshold(v, SEND), _threshold(v, FETCH)

        # The client's buffers: a shorter list leaves the end of a longer one.
        push, fetch = ((torch.zeros(P, dtype=torch.int32, device="cuda"),
                        torch.zeros(P, dtype=torch.float64, device="cuda"),
                        torch.zeros(1, dtype=torch.int64, device="cuda")) for _ in range(2))

        def listing(to, keep, values):
            at = keep.nonzero().reshape(-1)
            to[0][: at.numel()], to[1][: at.numel()], to[2][0] = at.int(), values[at].double(), at.numel()

        for t, copy in enumerate(copies):
            c, n = t % lam, t // lam
            now = x[3] if case["live"] else mine
            keep = _passes(_words(P, c, n, seed), now, cp)
            at = keep.nonzero().reshape(-1)
            y = [z[at] for z in x]
            _apply(rule, alpha, y, grads[t][at].double(), tau[t])
            for z, w in zip(x, y):
                z[at] = w
            got = _passes(_words(P, c | 1 << 31, n, seed), x[3] if case["live"] else mine, cf)
            copies[t] = torch.where(got, x[0], copy.double())
            listing(push, keep, grads[t])
            listing(fetch, got, x[0])
        if case["live"] and rule in ("fasgd", "fasgd-std"):
            # Decided on the server's rounded v: entries at the threshold may
            # go either way, which hardly moves theta but shifts the lists.
            return {"push": (None,) * 3, "fetch": (None,) * 3, "copies": [None] * len(copies), "theta": x[0]}
        return {"push": push, "fetch": fetch, "copies": copies, "theta": x[0]}
    if kind == "message":
        cp, cf = _mean_threshold(v, SEND), _mean_threshold(v, FETCH)

        def send(client, count, c):
            w = torch.tensor([_one_word(0xFFFFFFFF, client, count, seed)[0]])
            return bool(_passes(w, x[3].mean().reshape(1).cpu(), c))

        cache, sent, fetched = {}, [], []
        for t in range(len(copies)):
            c, n = t % lam, t // lam
            sent.append(send(c, n, cp))
            if sent[-1]:
                cache[c] = grads[t]
            g = cache[c].double() if c in cache else torch.zeros_like(x[0])
            _apply(rule, alpha, x, g, tau[t])
        for t, copy in enumerate(copies):
            fetched.append(send(t % lam | 1 << 31, t // lam, cf))
            copies[t] = x[0] if fetched[-1] else copy.double()
        flags = [torch.tensor(f, dtype=torch.int32) for f in (sent, fetched)]
        return {"sent": flags[0], "fetched": flags[1], "copies": copies, "theta": x[0]}
    sizes = _sizes(P, case["tensors"], seed)
    parts = [slice(int(e - s), int(e)) for s, e in zip(sizes, np.cumsum(sizes))]

    def decide(client, n, budget):
        vbar = np.array([float(x[3][p].mean()) for p in parts], np.float32)
        c = _smallest_c(sizes, vbar, budget, P)
        w = torch.tensor([_one_word((1 << 31) + t // 4, client, n, seed)[t % 4] for t in range(len(parts))])
        keep = _passes(w, torch.tensor(vbar), c).tolist()
        return [p for p, k in zip(parts, keep) if k], (
            torch.tensor(keep, dtype=torch.uint8), torch.tensor([c], dtype=torch.float64),
            torch.tensor([sum(int(s) for s, k in zip(sizes, keep) if k)]))

    for t, copy in enumerate(copies):
        c, n = t % lam, t // lam
        some, push = decide(c, n, int(SEND * P))
        for p in some:
            _apply(rule, alpha, [y[p] for y in x], grads[t][p].double(), tau[t])
        some, fetch = decide(c | 1 << 31, n, int(FETCH * P))
        copies[t] = copy.double()
        for p in some:
            copies[t][p] = x[0][p]
    return {"push": push, "fetch": fetch, "copies": copies, "theta": x[0]}
