"""Workloads of the DeTAG step library that its speed is followed on.

A case is one call a training program makes in its loop: it holds the state of all n workers ([n][d] float32 arrays on
one GPU) in a ``Session`` and advances it - one iteration with the library's synthetic gradient, with gradients the
program wrote itself, of the D-PSGD baseline, or several iterations in one call.  The listed sizes are the five
configurations of ``paper_2006_08085_b200.inputs``, the graphs of ``bench.py``'s extra legs and the paper's two
experiments; ``draw`` spreads over the same ranges.

Fields of a case: ``graph`` (ring, torus, regular4), ``n`` workers (``rows`` of the torus; 0 otherwise), ``d``
coordinates, ``K`` gossip rounds, ``eta`` momentum (negative: derived from the spectrum), ``mode`` (detag, external,
dpsgd), ``start`` (gradient at the model the step started from), ``steps`` per call, ``alpha``, ``sigma``, and the
range ``a_lo`` .. ``a_hi`` of the curvatures (log-uniform).
"""
import functools
import math

import numpy as np
import torch

from paper_2006_08085_b200 import binding as B
from paper_2006_08085_b200 import inputs
from paper_2006_08085_b200.session import Session

DEVICE = "cuda:0"
T0 = 3  # completed steps of the state a case starts from: the middle of a run


def _case(graph, n, d, K, eta=-1.0, mode="detag", start=False, steps=1, alpha=0.001, sigma=0.1, a_lo=0.5, a_hi=2.0,
          rows=0):
    return {"graph": graph, "n": n, "rows": rows, "d": d, "K": K, "eta": eta, "mode": mode, "start": start,
            "steps": steps, "alpha": alpha, "sigma": sigma, "a_lo": a_lo, "a_hi": a_hi}


def listed():
    return [
        # eight workers, a few thousand coordinates: a call is a launch
        dict(_case("ring", 8, 4096, 2, alpha=0.05), name="ring8"),
        # sixteen workers on a ring with a ResNet20-sized vector, the paper's second experiment: fits in L2
        dict(_case("ring", 16, 270_000, 4, alpha=0.01), name="ring16"),
        # the same experiment as it is run in earnest, gradients from back-propagation, the paper's tuned (eta, R)
        dict(_case("ring", 16, 270_000, 2, eta=0.2, mode="external", alpha=0.01), name="ring16 external"),
        # a LeNet-sized vector (odd length) on eight workers, twenty iterations per call
        dict(_case("ring", 8, 62_007, 2, eta=0.2, steps=20, alpha=0.05), name="ring8 twenty steps"),
        # plain D-PSGD (one gossip round, no momentum), the paper's main baseline, ragged length
        dict(_case("regular4", 32, 3_000_001, 1, eta=0.0, mode="dpsgd"), name="regular32 dpsgd"),
        # Algorithm 2 with its printed timing on a graph without structure between 32 and 64 workers, ragged length
        dict(_case("regular4", 48, 1_000_003, 4, start=True), name="regular48 printed"),
        # the large configurations: 8 x 8 torus, 256-worker ring, ill-conditioned 32-worker graph
        dict(_case("torus", 64, 11_200_000, 8, alpha=0.005, sigma=0.05, a_lo=0.1, a_hi=10.0, rows=8), name="torus64"),
        dict(_case("ring", 256, 1_000_000, 16, eta=0.2, alpha=0.002), name="ring256"),
        dict(_case("regular4", 32, 25_600_000, 6, a_lo=0.01, a_hi=100.0), name="regular32"),
        # the 256-worker ring at the phase length of Theorem 3, where every worker hears from every other
        dict(_case("ring", 256, 200_000, 196, alpha=0.002), name="ring256 theorem 3"),
        # graphs no structured kernel knows: 100 workers, and a 16 x 16 torus
        dict(_case("regular4", 100, 2_000_000, 6), name="regular100"),
        dict(_case("torus", 256, 500_000, 16, alpha=0.002, rows=16), name="torus256"),
    ]


def draw(rng):
    graph = rng.choice(["ring", "ring", "torus", "regular4", "regular4"])
    rows = 0
    if graph == "torus":
        rows, cols = rng.choice([4, 8, 8, rng.randint(3, 16)]), rng.choice([8, 8, rng.randint(3, 16)])
        n = rows * cols
    else:
        n = int(round(math.exp(rng.uniform(math.log(5), math.log(256)))))
        if graph == "ring" and n >= 64 and rng.random() < 0.5:
            n = n // 32 * 32
    K = rng.choice([1, 2, 3, 4, 6, 8, 12, 16])
    if graph == "ring" and n >= 64 and n % 32 == 0 and rng.random() < 0.3:
        K = rng.randint(17, 196)
    mode = rng.choice(["detag"] * 7 + ["external", "external", "dpsgd"])
    steps = rng.randint(2, 20) if mode == "detag" and n <= 32 and rng.random() < 0.25 else 1
    # worker-coordinates from the smallest configuration's to 2^27; the many-round cases stay below the largest listed one
    most = 27.0 if n <= 128 else 25.5
    wc = 2.0 ** rng.uniform(15.0, most)
    return _case(graph, n, max(17, int(wc / n) | 1 if rng.random() < 0.6 else int(wc / n)), K, eta=0.2, mode=mode,
                 start=mode == "detag" and rng.random() < 0.2, steps=steps,
                 alpha=rng.choice([0.001, 0.005, 0.01]), sigma=rng.choice([0.0, 0.05, 0.1, 0.1]),
                 a_lo=rng.choice([0.1, 0.5]), a_hi=rng.choice([2.0, 10.0]), rows=rows)


# ---------------------------------------------------------------------------------------------- graphs
def _edges(graph, n, rows):
    if graph == "ring":
        return {(i, (i + 1) % n) for i in range(n)}
    if graph == "torus":
        cols = n // rows
        return {(r * cols + c, q) for r in range(rows) for c in range(cols)
                for q in (((r + 1) % rows) * cols + c, r * cols + (c + 1) % cols)}
    rng = np.random.default_rng(1000 + n)  # two edge-disjoint Hamiltonian cycles

    def cycle():
        p = rng.permutation(n)
        return {frozenset((int(p[k]), int(p[(k + 1) % n]))) for k in range(n)}

    first, second = cycle(), cycle()
    while first & second:
        second = cycle()
    return {tuple(sorted(e)) for e in first | second}


@functools.lru_cache(maxsize=64)
def _matrix(graph, n, rows):
    """Metropolis weights of the graph, dense float64."""
    deg = np.zeros(n, dtype=np.int64)
    edges = _edges(graph, n, rows)
    for i, j in edges:
        deg[i] += 1
        deg[j] += 1
    m = np.zeros((n, n))
    for i, j in edges:
        m[i, j] = m[j, i] = 1.0 / (1.0 + max(deg[i], deg[j]))
    for i in range(n):
        m[i, i] = 1.0 - m[i].sum()
    return m


@functools.lru_cache(maxsize=64)
def _eta(graph, n, rows):
    ev = np.linalg.eigvalsh(_matrix(graph, n, rows))
    lam = max(abs(ev[0]), abs(ev[-2]))
    s = math.sqrt(1.0 - lam * lam)
    return (1.0 - s) / (1.0 + s)


def _momentum(case):
    return case["eta"] if case["eta"] >= 0.0 else _eta(case["graph"], case["n"], case["rows"])


# ---------------------------------------------------------------------------------------------- state
def _fill(case, seed, x, y, g, a, c, g_new):
    """A run's state: models near one another, per-worker targets, tracker and gradient of the current model."""
    gen = torch.Generator(device=x.device).manual_seed(seed)
    n = case["n"]
    mu = torch.randn((n, 1), generator=gen, device=x.device) * 2.0
    a.uniform_(math.log(case["a_lo"]), math.log(case["a_hi"]), generator=gen).exp_()
    c.normal_(generator=gen).add_(mu)
    x.normal_(generator=gen).mul_(0.1)
    x.add_(torch.randn((1, x.shape[1]), generator=gen, device=x.device))
    g.normal_(generator=gen).mul_(case["sigma"]).addcmul_(a, x).addcmul_(a, c, value=-1.0)
    y.copy_(g)
    if g_new is not None:
        g_new.normal_(generator=gen).mul_(0.1).add_(g)


def prepare(case, seed):
    m = inputs.csr_from_dense(_matrix(case["graph"], case["n"], case["rows"]))
    s = Session(m, case["d"], case["K"], _momentum(case), case["alpha"], sigma=case["sigma"], seed=seed % (1 << 62),
                device=DEVICE, external_gradient=case["mode"] == "external",
                algorithm=B.DETAG_ALGORITHM_DPSGD if case["mode"] == "dpsgd" else B.DETAG_ALGORITHM_DETAG,
                gradient_point=B.DETAG_GRADIENT_AT_PHASE_START if case["start"] else B.DETAG_GRADIENT_AT_NEW_MODEL)
    _fill(case, seed, s.x, s.y, s.g, s.a, s.c, s.g_new)
    B.detag_set_step(s.state, T0)
    return s, case


def run(state):
    s, case = state
    if case["steps"] > 1:
        s.step_many(case["steps"])
    else:
        s.step()
    d = case["d"]
    out = {"x": s.x[:, :d], "g": s.g[:, :d]}
    if case["mode"] != "dpsgd":
        out["y"] = s.y[:, :d]
    return out


def work(case):
    # x, y, g, a, c read, x, y, g written; caller-written gradients replace a, c; D-PSGD has no tracker
    per = {"detag": 32, "external": 28, "dpsgd": 24}[case["mode"]]
    wc = case["n"] * case["d"]
    nnz = int(np.count_nonzero(_matrix(case["graph"], case["n"], case["rows"])))
    arrays = 1 if case["mode"] == "dpsgd" else 2
    # the gossip rounds over the non-zero weights, or the product with their polynomial where that is less
    gossip = min(2.0 * nnz * case["K"] / case["n"], 2.0 * case["n"]) * arrays
    return {"bytes": float(per * wc), "flops": float(wc * case["steps"] * (gossip + 8))}


def tolerance(case):
    # float32 state, float64 sums, normals accurate to 1e-6.  Measured against exact(): 2.5e-8 to 1.4e-7 after one step
    # (the tracker, a difference of gradients, is the largest), 3e-7 after twenty
    return {"rel": 1.2e-6, "max": 4e-5} if case["steps"] > 1 else {"rel": 5e-7, "max": 2e-5}


# ---------------------------------------------------------------------------------------------- float64
def _normals(seed, t, n, j0, j1, device):
    """Philox4x32-10 with key (seed) and counter (j, j >> 32, i / 4, t), Box-Muller on 23-bit uniforms; [n][j1 - j0]."""
    mask = 0xFFFFFFFF
    j = torch.arange(j0, j1, dtype=torch.int64, device=device)[None, :]
    q = torch.arange((n + 3) // 4, dtype=torch.int64, device=device)[:, None]
    shape = (q.shape[0], j.shape[1])
    c0, c1 = (j & mask).expand(shape), (j >> 32).expand(shape)
    c2, c3 = q.expand(shape), torch.full(shape, t, dtype=torch.int64, device=device)
    k0, k1 = seed & mask, (seed >> 32) & mask
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((p1 >> 32) & mask) ^ c1 ^ k0, p1 & mask, ((p0 >> 32) & mask) ^ c3 ^ k1, p0 & mask
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    out = torch.empty((4 * shape[0], shape[1]), dtype=torch.float64, device=device)
    for p, (even, odd) in enumerate(((c0, c1), (c2, c3))):
        rad = torch.sqrt(-2.0 * torch.log(((even >> 9).double() + 0.5) * 2.0 ** -23))
        ang = (odd >> 9).double() * (2.0 * math.pi * 2.0 ** -23)
        out[2 * p::4] = rad * torch.cos(ang)
        out[2 * p + 1::4] = rad * torch.sin(ang)
    return out[:n]


def exact(case, seed):
    n, d, alpha, sigma = case["n"], case["d"], case["alpha"], case["sigma"]
    ld = (d + 3) // 4 * 4
    new = lambda: torch.empty((n, ld), dtype=torch.float32, device=DEVICE)  # noqa: E731
    x, y, g, a, c = new(), new(), new(), new(), new()
    g_new = new() if case["mode"] == "external" else None
    _fill(case, seed, x, y, g, a, c, g_new)
    m, eta = _matrix(case["graph"], n, case["rows"]), _momentum(case)
    prev = cur = np.eye(n)
    for _ in range(case["K"]):
        prev, cur = cur, (1.0 + eta) * (m @ cur) - eta * prev
    P = torch.from_numpy(cur).to(DEVICE)
    out = {k: torch.empty((n, d), dtype=torch.float64, device=DEVICE) for k in ("x", "y", "g")}
    chunk = max(1024, (1 << 25) // n)
    for j0 in range(0, d, chunk):
        j1 = min(d, j0 + chunk)
        xs, ys, gs, as_, cs = (v[:, j0:j1].double() for v in (x, y, g, a, c))
        for i in range(case["steps"]):
            if case["mode"] == "external":
                gn = g_new[:, j0:j1].double()
                ys = P @ (ys + gn - gs)
                xs, gs = P @ xs - alpha * ys, gn
                continue
            yt = P @ ys if case["mode"] == "detag" else gs
            xn = P @ xs - alpha * yt
            gn = as_ * ((xs if case["start"] else xn) - cs)
            if sigma != 0.0:
                gn = gn + sigma * _normals(seed % (1 << 62), T0 + 1 + i, n, j0, j1, DEVICE)
            xs, ys, gs = xn, yt + gn - gs, gn
        for k, v in (("x", xs), ("y", ys), ("g", gs)):
            out[k][:, j0:j1] = v
    if case["mode"] == "dpsgd":
        del out["y"]
    return out
