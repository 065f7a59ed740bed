"""Performance cases: what a pricing desk has this library do, through its public entry points.

Kinds of case
  price  a context that the program keeps (curve, volatilities, rule, strikes); one pass is
         ``simulate`` of one scheme and ``prices``
  model  the same with a fresh context in every pass: new market data is priced once
  batch  many uneven term structures in one launch (graph replay), then every instance's prices
  mlp    the learned drift (``LLL_MLP``): a kept context with its network, ``simulate`` and ``prices``
  grads  one training step's forward and backward pass on host feature rows: outputs, loss, gradients

Market data, strikes, rules, weights, feature rows and the Philox key are made from the seed.

The schemes run in FP32 (path state, weights, caplet payoffs); the C ABI hands the prices over in
double arrays.  They are kept here as FP32, the precision in which they are computed: FP32 input
constants alone put every scheme's prices 2e-7 to 7e-7 from 64 bits.  ``exact`` gives the 64-bit
values of the same schemes on the same Philox streams.

Whole training runs are not among the cases: hundreds of Adam steps on BF16 products turn one
changed rounding into other weights, so their results cannot be compared.  Training's work is
measured by its gradient pass.
"""
import dataclasses
import math

import numpy as np
import torch

from paper_1006_3340_gb300 import lll
from paper_1006_3340_gb300.workloads import Workload, batched_instances

# ---- the cases -------------------------------------------------------------


def listed():
    return [
        # a desk's smallest call: a short curve with fresh market data, priced at the money once
        dict(name="short_model", kind="model", family="short", N=10, s=10, Q=32, scheme="full",
             product="caplet", mapping="path", paths=4000),
        # the paper's numerical example at its own path count (heavy-tailed NIG, wide rule)
        dict(name="paper_picard", kind="price", family="heavy", N=10, s=5, Q=96, scheme="picard",
             product="caplet", mapping="path", paths=10000),
        # one quarterly 10-year curve at an intraday path budget, default launch
        dict(name="intraday_full", kind="price", family="quarterly", N=40, s=8, Q=64, scheme="full",
             product="caplet", mapping="path", paths=4096),
        # the same curve by Picard with its Euler steps in parallel
        dict(name="intraday_picard_step", kind="price", family="quarterly", N=40, s=8, Q=64, scheme="picard",
             product="caplet", mapping="step", paths=4096),
        # the end-of-day valuation: 2^20 paths of that curve (the benchmark's workload)
        dict(name="eod_picard", kind="price", family="quarterly", N=40, s=8, Q=64, scheme="picard",
             product="caplet", mapping="path", paths=1 << 20),
        # its co-terminal swaptions under the full scheme, with a ragged path count
        dict(name="eod_swaption_full", kind="price", family="quarterly", N=40, s=8, Q=64, scheme="full",
             product="swaption", mapping="path", paths=300007),
        # a 30-year curve under the full scheme
        dict(name="long_full", kind="price", family="long", N=120, s=4, Q=96, scheme="full",
             product="caplet", mapping="path", paths=1 << 17),
        # a portfolio of uneven term structures in one launch
        dict(name="portfolio_full", kind="batch", instances=32, scheme="full", paths=500000),
        # learned drift, one network row per rate and step (the benchmark's network)
        dict(name="mlp_rate", kind="mlp", family="quarterly", N=40, s=8, Q=64, hidden=128, layers=3, head=0,
             paths=1 << 15),
        # learned drift, vector head
        dict(name="mlp_vec", kind="mlp", family="quarterly", N=40, s=8, Q=64, hidden=128, layers=3, head=1,
             paths=1 << 18),
        # the 30-year curve's 256-wide vector head, ragged path count
        dict(name="mlp_wide", kind="mlp", family="long", N=120, s=4, Q=96, hidden=256, layers=4, head=1,
             paths=50000),
        # one training batch of the per-rate network, forward and backward
        dict(name="mlp_grads", kind="grads", family="quarterly", N=40, s=8, Q=64, hidden=128, layers=3,
             rows=8192),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["price", "price", "price", "price", "model", "batch", "mlp", "mlp", "grads"])
    if kind == "grads":
        return dict(kind="grads", family="quarterly", N=rng.randint(12, 60), s=8, Q=64, hidden=128,
                    layers=rng.randint(2, 4), rows=_log_int(rng, 512, 16384))
    if kind == "batch":
        return dict(kind="batch", instances=rng.randint(3, 32), scheme=rng.choice(["full", "picard"]),
                    paths=_log_int(rng, 30000, 500000))
    if kind == "mlp":
        shape = rng.choice(["rate", "vec", "wide"])
        if shape == "wide":
            return dict(kind="mlp", family="long", N=rng.randint(64, 120), s=4, Q=96, hidden=256,
                        layers=rng.randint(2, 4), head=1, paths=_log_int(rng, 2000, 50000))
        if shape == "vec":
            return dict(kind="mlp", family="quarterly", N=rng.randint(12, 48), s=8, Q=64, hidden=128, layers=3,
                        head=1, paths=_log_int(rng, 4096, 1 << 18))
        return dict(kind="mlp", family="quarterly", N=rng.randint(12, 40), s=8, Q=64, hidden=128,
                    layers=rng.randint(2, 3), head=0, paths=_log_int(rng, 2048, 1 << 15))
    family = rng.choice(["short", "heavy", "quarterly", "quarterly", "long"])
    N = {"short": (6, 12), "heavy": (8, 10), "quarterly": (20, 60), "long": (80, 120)}[family]
    N = rng.randint(*N)
    s = {"short": rng.randint(4, 10), "heavy": 5, "quarterly": 8, "long": 4}[family]
    Q = {"short": 32, "heavy": 96, "quarterly": 64, "long": 96}[family]
    scheme = rng.choice(["full", "picard"])
    mapping = rng.choice(["path", "path", "step"]) if scheme == "picard" else "path"
    units = s * N * (N - 1) // 2
    most = min(1 << 20, int(3.5e9 / units))
    if kind == "model":
        most = min(most, 40000)
    if mapping == "step":
        most = min(most, 8192)
    return dict(kind=kind, family=family, N=N, s=s, Q=Q, scheme=scheme, mapping=mapping,
                product="caplet" if mapping == "step" else rng.choice(["caplet", "caplet", "swaption"]),
                paths=_log_int(rng, 2000, most))


# ---- inputs ----------------------------------------------------------------


def _rule(alpha, beta, dbar, a, Q):
    """Q-point Gauss rule of x^2 nu(x) on [-a, a], nu the NIG Levy density (Golub-Welsch on a
    graded Gauss-Legendre mesh).  One rule serves a program as long as its NIG parameters stand."""
    t, w = np.polynomial.legendre.leggauss(24)
    edges = np.concatenate([[0.0], a * np.geomspace(1e-10, 1.0 / 16, 34)[:-1], np.linspace(a / 16, a, 16)])
    half, mid = 0.5 * np.diff(edges), 0.5 * (edges[1:] + edges[:-1])
    y = (mid[:, None] + half[:, None] * t).ravel()
    v = (half[:, None] * w).ravel()
    y, v = np.concatenate([-y[::-1], y]), np.concatenate([v[::-1], v])
    k1 = torch.special.scaled_modified_bessel_k1(torch.from_numpy(alpha * np.abs(y))).numpy()
    v = v * dbar * alpha / math.pi * np.abs(y) * np.exp(beta * y - alpha * np.abs(y)) * k1
    al, be = np.zeros(Q), np.zeros(Q)
    basis = [np.sqrt(v / v.sum())]
    for k in range(Q):
        u = y * basis[k]
        al[k] = u @ basis[k]
        B = np.array(basis)
        for _ in range(2):
            u = u - B.T @ (B @ u)
        be[k] = np.linalg.norm(u)
        basis.append(u / be[k])
    x, U = np.linalg.eigh(np.diag(al) + np.diag(be[:-1], 1) + np.diag(be[:-1], -1))
    return np.ascontiguousarray(x), np.ascontiguousarray(v.sum() * U[0] ** 2)


def _market(case, seed):
    """(workload, nodes, weights) of one term structure around its family's level."""
    rng = np.random.default_rng(seed)
    family, N, s = case["family"], case["N"], case["s"]
    delta = 0.5 if family in ("short", "heavy") else 0.25
    T = np.arange(N) * delta
    tau = T[None, 1:] - np.arange((N - 1) * s)[:, None] * (delta / s)
    a, offsets = 1.5, [-200, -100, 0, 100, 200]
    if family == "short":
        L0, lam, nig, offsets = np.full(N, 0.04), np.full_like(tau, 0.15), (18.0, -4.0, 1.0), [0]
    elif family == "heavy":
        L0 = 0.035 + 0.015 * T / 5.0
        lam, nig, a = np.broadcast_to(np.linspace(0.20, 0.12, N - 1), tau.shape), (1.5, 0.0, 1.5), 30.0
    elif family == "quarterly":
        L0, lam, nig = 0.03 + 0.01 * (1 - np.exp(-T / 3)), 0.1 + 0.08 * np.exp(-tau), (12.0, -3.0, 0.8)
    else:
        L0, lam, nig = 0.03 + 0.01 * (1 - np.exp(-T / 3)), 0.12 + 0.1 * np.exp(-0.5 * tau), (10.0, -2.5, 1.2)
        offsets = [-200, -150, -100, -50, 0, 50, 100, 150, 200]
    L0 = L0 * rng.uniform(0.9, 1.1) * np.exp(0.02 * rng.standard_normal(N))
    lam = np.ascontiguousarray(np.where(tau > -delta, lam, 0.0) * rng.uniform(0.9, 1.05))
    alpha, beta, dbar = nig[0] * rng.uniform(1.0, 1.05), nig[1] * rng.uniform(0.95, 1.05), nig[2] * rng.uniform(0.95, 1.05)
    strikes = np.maximum(L0[1:, None] + 1e-4 * np.asarray(offsets, dtype=np.float64)[None, :], 0.0)
    wl = Workload(family, N, delta, s, L0, lam, "nig", alpha=alpha, beta=beta, dbar=dbar, a=a, Q=case["Q"],
                  strikes=np.ascontiguousarray(strikes), paths=case.get("paths", 0), seed=int(rng.integers(1, 1 << 62)))
    return wl, *_rule(alpha, beta, dbar, a, case["Q"])


def _portfolio(case, seed):
    """The sizes, path budgets and NIG parameters are the portfolio's own; curves, volatilities
    and strikes move with the seed."""
    rng = np.random.default_rng(seed)
    members = []
    for wl in batched_instances(n_inst=case["instances"], total_paths=case["paths"], seed=case["instances"]):
        up = rng.uniform(0.9, 1.1) * np.exp(0.02 * rng.standard_normal(wl.N))
        wl = dataclasses.replace(wl, L0=wl.L0 * up, strikes=wl.strikes * up[1:, None], lam=wl.lam * rng.uniform(0.9, 1.05))
        members.append((wl, *_rule(wl.alpha, wl.beta, wl.dbar, wl.a, wl.Q)))
    return members


def _bf16(v):
    return torch.from_numpy(np.ascontiguousarray(v, dtype=np.float32)).bfloat16().float().numpy()


def _network(case, wl, seed):
    """Weights of a trained network's size ((W, b) pairs, W already BF16 numbers) and the five
    feature and target scales (time, rate index, volatility, log-rate, compensator)."""
    rng = np.random.default_rng([seed, 1])
    head = case.get("head", 0)
    outputs = (wl.n + 15) // 16 * 16 if head else 1
    sizes = [1 + wl.N if head else 3 + wl.N] + [case["hidden"]] * case["layers"] + [outputs]
    net = [(_bf16(rng.uniform(-1, 1, (o, i)) * math.sqrt((6.0 if k < case["layers"] else 3.0) / i)),
            rng.normal(scale=0.05, size=o).astype(np.float32)) for k, (i, o) in enumerate(zip(sizes[:-1], sizes[1:]))]
    scales = np.array([1.0 / (wl.N * wl.delta), 1.0 / wl.n, 1.0 / wl.lam.max(), 4.0, 1.5e-4], dtype=np.float32)
    return net, scales


def _rows(case, wl, seed):
    """A training batch: feature rows (t, i, lambda, log-rate offsets) and unit-RMS targets."""
    rng = np.random.default_rng([seed, 2])
    rows = case["rows"]
    i = rng.integers(1, wl.n + 1, rows)
    k = (rng.random(rows) * i * wl.s).astype(np.int64)
    t = k * wl.h
    u = rng.normal(scale=0.15, size=(rows, wl.N)) * np.sqrt(t)[:, None] * 4.0
    u[:, 0] = 0.0
    x = np.concatenate([(t / (wl.N * wl.delta))[:, None], (i / wl.n)[:, None],
                        (wl.lam[k, i - 1] / wl.lam.max())[:, None], u], axis=1)
    return _bf16(x), rng.standard_normal(rows).astype(np.float32)


def _pack(net, offsets, count, in_pad):
    flat = np.zeros(count, dtype=np.float32)
    for k, (W, b) in enumerate(net):
        if k == 0:
            W = np.concatenate([W, np.zeros((W.shape[0], in_pad - W.shape[1]), np.float32)], axis=1)
        flat[offsets[2 * k]: offsets[2 * k] + W.size] = W.ravel()
        flat[offsets[2 * k + 1]: offsets[2 * k + 1] + b.size] = b
    return flat


class _Batch:
    def __init__(self, members):
        self.members = [wl for wl, _, _ in members]
        self.handle, self.keep = lll.lll_batch_init(members)
        lll.lll_batch_use_graph(self.handle, True)

    def __del__(self):
        lll.lll_batch_destroy(self.handle)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return dict(case=case, batch=_Batch(_portfolio(case, seed)), seed=int(seed) + 12345)
    wl, x, W = _market(case, seed)
    if kind == "model":
        return dict(case=case, wl=wl, x=x, W=W)
    sim = lll.LevyLibor(wl, x, W)
    state = dict(case=case, wl=wl, sim=sim)
    if kind == "price":
        sim.set_product(case["product"])
        sim.set_mapping(case["mapping"])
        return state
    net, scales = _network(case, wl, seed)
    lll.lll_mlp_init(sim.ctx, case["hidden"], case["layers"], seed=1, head=case.get("head", 0))
    count, _, in_pad, offsets = lll.lll_mlp_layout(sim.ctx, case["layers"])
    lll.lll_mlp_params(sim.ctx, 1, _pack(net, offsets, count, in_pad), scales=scales)
    if kind == "grads":
        state["xy"] = _rows(case, wl, seed)
        state["count"] = count
    return state


# ---- one pass --------------------------------------------------------------


def _priced(p, se):
    return dict(prices=p.astype(np.float32), stderr=se.astype(np.float32))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batch":
        b = state["batch"]
        lll.lll_batch_simulate(b.handle, lll.SCHEMES[case["scheme"]], state["seed"])
        return [_priced(*lll.lll_batch_prices(b.handle, q, wl.n, wl.strikes.shape[1]))
                for q, wl in enumerate(b.members)]
    if kind == "grads":
        out, g, loss = lll.lll_mlp_eval(state["sim"].ctx, *state["xy"], state["count"], want_grads=True)
        return dict(out=out, grads=g, loss=np.float32(loss))
    if kind == "model":
        sim = lll.LevyLibor(state["wl"], state["x"], state["W"])
        sim.set_product(case["product"])
        sim.set_mapping(case["mapping"])
    else:
        sim = state["sim"]
    sim.simulate("mlp" if kind == "mlp" else case["scheme"])
    result = _priced(*sim.prices())
    if kind == "model":
        sim.close()
    return result


# ---- what a pass cannot do without -----------------------------------------


def _mlp_flops(case, N):
    n, H, L = N - 1, case["hidden"], case["layers"]
    head = case.get("head", 0)
    return 2.0 * ((1 + N if head else 3 + N) * H + (L - 1) * H * H + H * (n if head else 1))


def _path_work(N, s, ns, paths):
    """Bytes: curve, volatility table, strikes and rule in, prices out.  Operations per path: a step
    draws its increment (a counter-based word, Box-Muller, the inverse Gaussian root: about 120);
    a live rate's step costs its weight 1/(1 + e^-x), the Euler update (about 10) and the drift
    integral, whose integrand is smooth enough for a rule of eight nodes on these ranges, however
    many nodes state the measure (8 x 3); a payoff costs about 10 per rate alive at its date."""
    n = N - 1
    units = s * n * (n + 1) / 2
    return (dict(bytes=8.0 * (N + n * s * n + 3 * n * ns + 128),
                 flops=paths * (120.0 * n * s + 34.0 * units + 10.0 * (n * (n + 1) / 2 + n * ns))),
            units * paths, float(n * s) * paths)


def work(case):
    if case["kind"] == "batch":
        wls = batched_instances(n_inst=case["instances"], total_paths=case["paths"], seed=case["instances"])
        got = [_path_work(wl.N, wl.s, wl.strikes.shape[1], wl.paths)[0] for wl in wls]
        return {k: sum(w[k] for w in got) for k in ("bytes", "flops")}
    N = case["N"]
    if case["kind"] == "grads":
        per = _mlp_flops(case, N)
        params = per / 2 + case["layers"] * case["hidden"] + 1
        return dict(bytes=4.0 * (case["rows"] * (N + 5) + 2 * params), flops=3.0 * per * case["rows"])
    ns = {"short": 1, "heavy": 5, "quarterly": 5, "long": 9}[case["family"]]
    w, units, steps = _path_work(N, case["s"], ns, case["paths"])
    if case["kind"] == "mlp":
        w["flops"] += _mlp_flops(case, N) * (steps if case["head"] else units) - 24.0 * units
    return w


# ---- the same in 64 bits ---------------------------------------------------


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _philox(k, inst, path, key):
    """Philox-4x32-10 words 0..2 for counters (k, inst, path lo, path hi), 64-bit integer tensors."""
    mask = 0xFFFFFFFF

    def mul(c, v):  # 32 x 32 bits: (high, low)
        return ((c * (v >> 16) + ((c * (v & 0xFFFF)) >> 16)) >> 16) & mask, (c * v) & mask

    c = [k, torch.full_like(k, inst), path & mask, path >> 32]
    k0, k1 = key & mask, (key >> 32) & mask
    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c[:3]


def _increments(wl, paths, inst, key):
    """NIG increments [S, paths] by Michael, Schucany and Haas from three uniforms a step."""
    k = torch.arange(wl.steps, device=paths.device)[:, None].expand(-1, len(paths)).contiguous()
    u0, u1, u2 = ((w >> 9).double() / 8388608.0 + 1.0 / 16777216.0
                  for w in _philox(k, inst, paths[None, :].expand_as(k).contiguous(), key))
    r = torch.sqrt(-2.0 * torch.log(u0))
    nu, z = (r * torch.cos(2 * math.pi * u1)) ** 2, r * torch.sin(2 * math.pi * u1)
    g = math.sqrt(wl.alpha ** 2 - wl.beta ** 2)
    m, l = wl.dbar * wl.h / g, (wl.dbar * wl.h) ** 2
    big = m + m * m * nu / (2 * l) + m / (2 * l) * torch.sqrt(4 * m * l * nu + (m * nu) ** 2)
    small = m * m / big
    V = torch.where(u2 <= m / (m + small), small, big)
    return wl.beta * V + torch.sqrt(V) * z - wl.dbar * wl.beta / g * wl.h


def _exact_prices(wl, x, W, scheme, product="caplet", inst=0, seed=None, net=None, scales=None, head=0):
    dev = _device()
    n, s, S, h = wl.n, wl.s, wl.steps, wl.h
    f8 = lambda v: torch.from_numpy(np.ascontiguousarray(v, dtype=np.float64)).to(dev)  # noqa: E731
    xs, c = f8(x), f8(W / x ** 2)
    lam, L0 = f8(wl.lam), f8(wl.L0[1:])
    logL0 = torch.log(L0)[:, None]
    BN = float(np.prod(1.0 / (1.0 + wl.delta * wl.L0)))
    if net is not None:
        net = [(f8(A), f8(b)) for A, b in net]
        sc = [float(v) for v in scales]

    def drift(k, live, w):
        """Compensators A [live, paths] of the rates n, n-1, .., imin, w [live, paths] likewise."""
        lk = lam[k, live]
        E = torch.expm1(lk[:, None] * xs)
        C = (c * (E - lk[:, None] * xs)).sum(1)
        A = C[:, None].expand(-1, w.shape[1]).clone()
        if len(live) > 1:
            P = torch.addcmul(torch.ones((), dtype=torch.float64, device=dev), w[:-1, :, None], E[:-1, None, :])
            P = torch.cumprod(P, 0, out=P).sub_(1.0)
            A[1:] += torch.matmul(P, (E * c)[1:, :, None])[:, :, 0]
        return A

    def learned(k, live, U):
        paths = U.shape[1]
        lk = lam[k, live]
        E = torch.expm1(lk[:, None] * xs)
        C = (c * (E - lk[:, None] * xs)).sum(1)
        u = torch.zeros((paths, wl.N), dtype=torch.float64, device=dev)
        u[:, 1:] = U.T * sc[3]
        (W0, b0), rest = net[0], net[1:]
        if head:
            z = u @ W0[:, 1:].T + (W0[:, 0] * (k * h * sc[0]) + b0)
        else:
            own = torch.stack([torch.full_like(lk, k * h * sc[0]), (live + 1).double() * sc[1], lk * sc[2]], 1)
            z = (u @ W0[:, 3:].T)[None] + (own @ W0[:, :3].T + b0)[:, None, :]
        for A, b in rest:
            z = torch.nn.functional.silu(z) @ A.T + b
        f = z[:, live].T if head else z[:, :, 0]
        return C[:, None] + sc[4] * f

    D0 = torch.zeros((S + 1, n), dtype=torch.float64, device=dev)
    if scheme == "picard":  # running integral of the drift at the initial curve
        w0 = wl.delta * L0 / (1 + wl.delta * L0)
        for k in range(S):
            live = torch.arange(n - 1, k // s - 1, -1, device=dev)
            D0[k + 1] = D0[k]
            D0[k + 1, live] -= drift(k, live, w0[live, None])[:, 0] * h
    s1 = torch.zeros((n, wl.strikes.shape[1]), dtype=torch.float64, device=dev)
    s2 = torch.zeros_like(s1)
    strikes = f8(wl.strikes)
    if net is None:
        chunk = max(256, (1 << 25) // (n * len(x)))
    else:
        chunk = max(256, (1 << 28) // (net[0][0].shape[0] * (1 if head else n)))
    for first in range(0, wl.paths, chunk):
        p = torch.arange(first, min(first + chunk, wl.paths), device=dev)
        dH = _increments(wl, p, inst, wl.seed if seed is None else seed)
        Z = torch.zeros((n, len(p)), dtype=torch.float64, device=dev)
        Y = torch.zeros_like(Z)
        for k in range(S):
            live = torch.arange(n - 1, k // s - 1, -1, device=dev)
            if net is not None:
                A = learned(k, live, Z)
            else:
                at = logL0[live] + (D0[k, live, None] + Y[live] if scheme == "picard" else Z[live])
                A = drift(k, live, torch.sigmoid(at + math.log(wl.delta)))
            jump = lam[k, live, None] * dH[k]
            Z[live] += jump - A * h
            Y[live] += jump
            if (k + 1) % s == 0:
                m = k // s  # rate index m fixes at T_{m+1}
                L = torch.exp(logL0[m:] + Z[m:])
                B = torch.flip(torch.cumprod(torch.flip(1 + wl.delta * L, [0]), 0), [0])
                if product == "caplet":
                    P = B[1] if m + 1 < n else torch.ones_like(B[0])
                    v = wl.delta * BN * P[:, None] * torch.clamp(L[0][:, None] - strikes[m], min=0.0)
                else:
                    v = BN * torch.clamp((B[0] - 1)[:, None] - strikes[m] * wl.delta * (1 + B[1:].sum(0))[:, None], min=0.0)
                s1[m] += v.sum(0)
                s2[m] += (v * v).sum(0)
    P = float(wl.paths)
    mean = s1 / P
    var = torch.clamp(s2 / P - mean * mean, min=0.0) * P / max(P - 1.0, 1.0)
    return dict(prices=mean.cpu().numpy(), stderr=torch.sqrt(var / P).cpu().numpy())


def _exact_grads(case, wl, seed):
    net, _ = _network(case, wl, seed)
    x, y = _rows(case, wl, seed)
    ps = [[torch.from_numpy(v.astype(np.float64)).requires_grad_() for v in pair] for pair in net]
    h = torch.from_numpy(x.astype(np.float64))
    for k, (A, b) in enumerate(ps):
        h = (torch.nn.functional.silu(h) if k else h) @ A.T + b
    loss = ((h[:, 0] - torch.from_numpy(y.astype(np.float64))) ** 2).mean()
    loss.backward()
    in_pad = (wl.N + 3 + 15) // 16 * 16
    offsets, at = [], 0
    for k, (A, b) in enumerate(ps):  # the flat layout: W, b by layers, each on a multiple of 8
        for size in (A.shape[0] * (in_pad if k == 0 else A.shape[1]), b.numel()):
            offsets.append(at)
            at = (at + size + 7) // 8 * 8
    grads = np.zeros(at)
    for k, (A, b) in enumerate(ps):
        G = np.zeros((A.shape[0], in_pad)) if k == 0 else np.zeros(tuple(A.shape))
        G[:, : A.shape[1]] = A.grad.numpy()
        grads[offsets[2 * k]: offsets[2 * k] + G.size] = G.ravel()
        grads[offsets[2 * k + 1]: offsets[2 * k + 1] + b.numel()] = b.grad.numpy()
    return dict(out=h[:, 0].detach().numpy(), grads=grads, loss=float(loss))


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return [_exact_prices(*m, case["scheme"], inst=q, seed=int(seed) + 12345)
                for q, m in enumerate(_portfolio(case, seed))]
    wl, x, W = _market(case, seed)
    if kind == "grads":
        return _exact_grads(case, wl, seed)
    if kind == "mlp":
        if work(case)["flops"] > 2e13:  # too long in 64 bits
            return None
        net, scales = _network(case, wl, seed)
        return _exact_prices(wl, x, W, "full", net=net, scales=scales, head=case["head"])
    return _exact_prices(wl, x, W, case["scheme"], case["product"])
