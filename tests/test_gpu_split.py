"""The polynomial on the integer tensor path (48 < n <= 256; the cases of 33 to 48 workers run on step_dense.cu and hold it to the
same): tile edges, block structures, modes, and the coordinates it
contracts in float64 instead (an output may read nothing near the largest operand, infinities, NaN)."""
import numpy as np
import pytest

from oracle import detag_oracle as orc
from paper_2006_08085_b200 import binding as B
from paper_2006_08085_b200 import build, inputs
from paper_2006_08085_b200.session import Session
from parity import HALF_ULP32, one_step_from_rounded_state, oracle_problem, worst_ratio

pytestmark = pytest.mark.gpu

SLABS = 64 * 148  # one slab of 64 coordinates per block


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def _graph(kind, n):
    if kind == "ring":
        return inputs.metropolis_weights(inputs.ring_graph(n))
    if kind == "torus":
        return inputs.metropolis_weights(inputs.torus_graph(n // 16, 16))
    if kind == "path":
        return inputs.metropolis_weights(inputs.path_graph(n))
    if kind == "directed":
        return inputs.directed_cycle_blend(n, 0.4, 0.35)
    return inputs.metropolis_weights(inputs.random_regular4_graph(n, n))


def _data(n, d, seed):
    rng = np.random.default_rng(seed)
    a = rng.uniform(0.5, 2.0, (n, d)).astype(np.float32)
    c = (0.1 * (rng.standard_normal((n, d)) + np.arange(n)[:, None] - n / 2)).astype(np.float32)
    return a, c, rng.standard_normal((n, d)).astype(np.float32)


# n: one worker beyond a block, whole blocks, a last unit of one worker, an odd number of half chunks; d: below, at and
# beyond a slab, tails of 1 .. 3 columns, several slabs per block of the grid
@pytest.mark.parametrize("n,d,K,kind,at_start", [
    (33, 1, 2, "regular4", False), (48, 63, 3, "regular4", True), (50, 1, 2, "regular4", False), (57, 63, 3, "regular4", True), (49, 2 * SLABS + 66, 2, "path", False),
    (64, 64, 5, "ring", False), (65, 65, 3, "directed", True), (81, 5 * SLABS + 3, 4, "regular4", False),
    (113, 130, 6, "regular4", False), (128, 3 * SLABS + 31, 9, "regular4", True), (160, 97, 12, "ring", False),
    (224, 2 * SLABS + 2, 40, "ring", False), (256, 131, 16, "torus", True), (256, 3 * SLABS + 7, 16, "torus", False),
    (256, 2 * SLABS + 65, 16, "ring", False)])
def test_one_step_against_the_oracle(n, d, K, kind, at_start):
    m = _graph(kind, n)
    eta = 0.3
    cols = np.unique(np.concatenate([np.arange(min(d, 70)), np.arange(max(0, d - 70), d),
                                     np.random.default_rng(1).integers(0, d, 60)]))
    a, c, x0 = _data(n, d, n + d)
    # the oracle on a sample of the columns (the step never mixes them), the noise index of each being its column
    ref = {}
    for lo, hi in _runs(cols):
        p = oracle_problem(m, K, eta, 0.02, a[:, lo:hi], c[:, lo:hi], 0.1, 11, lo)
        if at_start:
            s = orc.PhaseState(x0[:, lo:hi].astype(np.float64), a[:, lo:hi].astype(np.float64),
                               c[:, lo:hi].astype(np.float64), 0)
            out = orc.phase_as_printed(p, s)
            g = orc.stochastic_gradient(p, s.x, 1)
            ref[lo, hi] = (out.x, None, g, out.y)
        else:
            ref[lo, hi] = one_step_from_rounded_state(p, x0[:, lo:hi])
    with Session(m, d, K, eta, 0.02, a, c, x0, 0.1, 11, observe_gossip=True,
                 gradient_point=int(at_start)) as s:
        if at_start:  # any tracker and gradient will do: the objective's arrays
            s.upload("y", a)
            s.upload("g", c)
            B.detag_set_step(s.state, 0)
        else:
            s.init()
        s.step()
        s.status()
        got = {k: s.download(k) for k in ("x", "y_gossip", "g", "y")}
    for (lo, hi), want in ref.items():
        x, yg, g, yf = want if at_start else want[1]
        cut = {k: v[:, lo:hi] for k, v in got.items()}
        assert worst_ratio(cut["x"], x) <= 1.0, (lo, "x")
        assert worst_ratio(cut["g"], g) <= 1.0, (lo, "g")
        assert worst_ratio(cut["y"], yf, extra=HALF_ULP32 * np.abs(g)) <= 1.0, (lo, "y")
        if yg is not None:
            assert worst_ratio(cut["y_gossip"], yg) <= 1.0, (lo, "y_gossip")


def _runs(cols):
    """Consecutive stretches [lo, hi) of a sorted column list."""
    cuts = np.flatnonzero(np.diff(cols) > 1) + 1
    return [(int(r[0]), int(r[-1]) + 1) for r in np.split(cols, cuts)]


@pytest.mark.parametrize("n,kind,K", [(40, "ring", 2), (56, "ring", 2), (100, "regular4", 2), (100, "regular4", 8), (256, "ring", 9)])
def test_values_far_apart_keep_their_precision(n, kind, K):
    """A few neighbouring workers a million times larger than the rest: results out of their reach must not inherit their
    scale.  A float64 sum rounded once to float32 is off by half an ulp, 2^-24 of itself, and that is all in those columns
    if the polynomial has entries below 2^-8 of their row's largest.  Elsewhere the bound allows 2^-24.4 of the largest
    operand times the row's largest entry, far more than the kernel's digits leave out (2^-37)."""
    d, eta = 200, 0.2
    m = _graph(kind, n)
    P = _polynomial(m, K, eta)
    rng = np.random.default_rng(n)
    x = rng.standard_normal((n, d)).astype(np.float32)
    x[:3, ::7] *= 1e6
    x[:, 5] = 0.0
    x[:, 12] = 0.0
    x[7, 12] = 3e-39  # the only value of its column: below the range of the scale
    zero = np.zeros((n, d), np.float32)
    with Session(m, d, K, eta, 0.0, zero, zero, x) as s:
        s.step()
        s.status()
        got = s.download("x").astype(np.float64)
    x = x.astype(np.float64)
    top = np.abs(P).max(axis=1, keepdims=True)
    bound = 2.0 ** -24 * np.abs(P @ x) + 2.0 ** -45 * (np.abs(P) @ np.abs(x)) + 1e-45
    split = np.ones(d, bool)
    split[::7] = not (np.abs(P) < top / 256).any()
    bound += np.where(split, 2.0 ** -24.4 * top * np.abs(x).max(axis=0), 0.0)
    assert (np.abs(got - P @ x) <= bound).all()
    assert (got[:, 5] == 0.0).all()


def _unequal(pattern, n, d, rng):
    z = rng.standard_normal((n, d))
    if pattern == "one larger":
        z[n // 3] *= 2.0 ** 9
    elif pattern == "every eighth":
        z[::8] *= 10.0 ** rng.integers(3, 9, d)
    elif pattern == "all but the last":
        z[:n - n % 8 - (n % 8 == 0) * 4] *= 1e6
    elif pattern == "sorted":
        z *= (10.0 ** np.linspace(-2, 2, n))[:, None]
    elif pattern == "log-uniform":
        z *= 10.0 ** rng.uniform(-2, 2, (n, d))
    elif pattern == "one alone":
        z[np.arange(n) != n // 2] = 0.0
    elif pattern == "consensus":
        z = z[:1] + 1e-6 * z
    return z.astype(np.float32)


@pytest.mark.parametrize("kind,n", [("ring", 36), ("regular4", 48), ("ring", 52), ("regular4", 60), ("ring", 100), ("regular4", 100), ("directed", 128),
                                    ("ring", 224), ("torus", 256)])
@pytest.mark.parametrize("K", [1, 2, 6, 16])
def test_every_result_is_as_precise_as_what_it_reads(kind, n, K):
    """P z per element, model and tracker, against float64: half an ulp of the stored value, 2^-24 |P z|, and as much again
    for the sum, 2^-24 |P| |z| - the magnitudes that this very output reads, whatever the other workers hold."""
    d, eta = 150, 0.2
    m = _graph(kind, n)
    P = _polynomial(m, K, eta)
    rng = np.random.default_rng(n * 31 + K)
    zero = np.zeros((n, d), np.float32)
    patterns = ["alike", "one larger", "every eighth", "all but the last", "sorted", "log-uniform", "one alone", "consensus"]
    with Session(m, d, K, eta, 0.0, zero, zero, zero) as s:
        for k, pattern in enumerate(patterns):
            state = {"x": _unequal(pattern, n, d, rng), "y": _unequal(patterns[k - 1], n, d, rng)}
            s.upload("g", zero)
            for name, v in state.items():
                s.upload(name, v)
            B.detag_set_step(s.state, 0)
            s.step()
            s.status()
            for name, v in state.items():
                got, z = s.download(name).astype(np.float64), v.astype(np.float64)
                bound = 2.0 ** -24 * (np.abs(P @ z) + np.abs(P) @ np.abs(z)) + 1e-45
                worst = (np.abs(got - P @ z) / bound).max()
                assert worst <= 1.0, (pattern if name == "x" else patterns[k - 1], name, worst)


@pytest.mark.parametrize("n,bad", [(48, np.inf), (60, np.inf), (100, np.nan), (256, -np.inf)])
def test_what_is_not_finite_stays_in_reach(n, bad):
    d, K, eta = 130, 2, 0.2
    m = _graph("ring", n)
    P = _polynomial(m, K, eta)
    x = np.random.default_rng(n).standard_normal((n, d)).astype(np.float32)
    x[9, 70] = bad
    zero = np.zeros((n, d), np.float32)
    with Session(m, d, K, eta, 0.0, zero, zero, x) as s:
        s.step()
        s.status()
        got = s.download("x")
    reached = P[:, 9] != 0.0
    assert not np.isfinite(got[reached, 70]).any()
    keep = np.ones((n, d), bool)
    keep[reached, 70] = False
    x[9, 70] = 0.0
    assert worst_ratio(got[keep], (P @ x.astype(np.float64))[keep]) <= 1.0


@pytest.mark.parametrize("n,K,worker", [(256, 34, 31), (256, 33, 224), (128, 35, 31)])
def test_faint_entries_reach_as_far_as_the_polynomial(n, K, worker):
    """Entries of P far below the largest of their row (1e-10 .. 1e-16 of it, whole blocks of them): an infinity travels
    through them, and so does an operand large enough to make up for them."""
    d, eta = 65, 0.2
    m = _graph("ring", n)
    P = _polynomial(m, K, eta)
    x = np.random.default_rng(n + K).standard_normal((n, d)).astype(np.float32)
    x[worker, 3] = np.inf
    x[worker, 40] = 1e20
    zero = np.zeros((n, d), np.float32)
    with Session(m, d, K, eta, 0.0, zero, zero, x) as s:
        s.step()
        s.status()
        got = s.download("x")
    reached = P[:, worker] != 0.0
    faint = np.abs(P[:, worker]) < 2.0 ** -32 * np.abs(P).max()
    assert (reached & faint).any()
    assert not np.isfinite(got[reached, 3]).any() and np.isfinite(got[~reached, 3]).all()
    x = x.astype(np.float64)
    bound = 2.0 ** -24 * np.abs(P @ x[:, 40]) + 2.0 ** -45 * (np.abs(P) @ np.abs(x[:, 40]))
    assert (np.abs(got[:, 40] - P @ x[:, 40]) <= bound).all()


def _polynomial(m, K, eta):
    w = m.to_dense()
    prev = cur = np.eye(m.n)
    for _ in range(K):
        prev, cur = cur, (1.0 + eta) * w @ cur - eta * prev
    return cur


@pytest.mark.parametrize("n,d", [(50, 131), (70, 67), (96, 2 * SLABS + 5), (256, 129)])
def test_dpsgd(n, d):
    m = _graph("ring", n)
    a, c, x0 = _data(n, d, n)
    K, eta, alpha = 3, 0.2, 0.05
    with Session(m, d, K, eta, alpha, a, c, x0, 0.1, 3, algorithm=B.DETAG_ALGORITHM_DPSGD) as s:
        s.upload("g", c)
        s.upload("y", a)
        B.detag_set_step(s.state, 0)
        s.step()
        s.status()
        x, g, y = (s.download(k) for k in ("x", "g", "y"))
    want = _polynomial(m, K, eta) @ x0.astype(np.float64) - alpha * c
    assert worst_ratio(x, want) <= 1.0
    for lo, hi in ((0, min(d, 100)), (max(0, d - 100), d)):
        p = oracle_problem(m, K, eta, alpha, a[:, lo:hi], c[:, lo:hi], 0.1, 3, lo)
        assert worst_ratio(g[:, lo:hi], orc.stochastic_gradient(p, want[:, lo:hi], 1)) <= 1.0
    assert np.array_equal(y, a)  # no tracker: untouched


# What the dispatch leaves to step_split.cu: the DeTAG step of 65 to 96 workers and D-PSGD of sparse polynomials, not the shortest, long vectors of 49 to 64
# (two slabs' digits), the longest of 97 to 128 with the printed timing, block-circulant matrices beyond 128 workers with more than one (dense polynomials: thirteen, D-PSGD three) chunk per block
KEPT = [(72, "regular4", 4_003, 2, "detag"), (90, "path", 4_003, 6, "start"), (96, "regular4", SLABS + 33, 16, "detag"), (81, "regular4", 3_600, 1, "detag"), (128, "regular4", 890_371, 3, "start"),
        (49, "path", 152_001, 2, "detag"), (60, "regular4", 160_003, 6, "start"), (60, "ring", 160_001, 3, "dpsgd"), (90, "regular4", 303_202, 2, "dpsgd"),
        (160, "ring", 5_003, 20, "detag"), (224, "ring", 5_001, 17, "start"), (256, "ring", 190_002, 34, "detag"), (256, "torus", 5_003, 2, "detag"),
        (256, "torus", 19_001, 3, "dpsgd"), (256, "torus", 190_001, 16, "detag")]


@pytest.mark.parametrize("n,kind,d,K,mode", KEPT)
def test_every_result_is_as_precise_as_what_it_reads_at_lengths_that_this_kernel_keeps(n, kind, d, K, mode):
    patterns_side_by_side(n, kind, d, K, mode, "step_split")


def patterns_side_by_side(n, kind, d, K, mode, kernel):
    """As above, every column of the model and of the tracker; an infinity in one column and a NaN in another reach as far as the polynomial."""
    eta, wide = 0.2, 1997
    m = _graph(kind, n)
    P = _polynomial(m, K, eta)
    rng = np.random.default_rng(n + d)
    patterns = ["alike", "one larger", "every eighth", "all but the last", "sorted", "log-uniform", "one alone", "consensus"]
    # a block of columns over and over: patterns side by side, so that one slab holds coordinates of both kinds
    blocks = {}
    for shift, name in enumerate(("x", "y")):
        z = np.empty((n, wide), np.float32)
        for k, pattern in enumerate(patterns):
            at = (np.arange(wide) + 3 * shift) % 8 == k
            z[:, at] = _unequal(pattern, n, int(at.sum()), rng)
        blocks[name] = z
    state = {k: np.ascontiguousarray(np.tile(z, -(-d // wide))[:, :d]) for k, z in blocks.items()}
    bad = {"x": (d // 2 + 1, np.inf), "y": (d - 2, np.nan)}
    for name, (col, v) in bad.items():
        state[name][9, col] = v
    zero = np.zeros((n, d), np.float32)
    with Session(m, d, K, eta, 0.0, zero, zero, zero, gradient_point=int(mode == "start"), algorithm=int(mode == "dpsgd")) as s:
        for name, v in state.items():
            s.upload(name, v)
        s.step()
        s.status()
        assert B.detag_debug_kernel(s.state) == kernel
        got = {k: s.download(k) for k in ("x", "y")}
    reached = P[:, 9] != 0.0
    if mode == "dpsgd":
        assert np.array_equal(got.pop("y"), state["y"], equal_nan=True)  # no tracker: untouched
    for name, have in got.items():
        z = blocks[name].astype(np.float64)
        want = P @ z
        bound = 2.0 ** -24 * (np.abs(want) + np.abs(P) @ np.abs(z)) + 1e-45
        for lo in range(0, d, wide):
            cut = have[:, lo:lo + wide].astype(np.float64)
            keep = np.ones(cut.shape, bool)
            for other, (col, _) in bad.items():
                if lo <= col < lo + wide:  # x' = P x - 0 * P y, y' = P y + 0 * x'
                    assert other != name or not np.isfinite(cut[reached, col - lo]).any()
                    keep[reached, col - lo] = False
            w = cut.shape[1]
            assert ((np.abs(cut - want[:, :w]) <= bound[:, :w]) | ~keep).all(), (name, lo)


@pytest.mark.parametrize("n,kind,d,K,mode", [(72, "regular4", 2 * SLABS + 5, 3, "detag"), (60, "regular4", 17 * SLABS + 5, 3, "start"),
                                             (90, "regular4", 303_202, 2, "dpsgd"), (256, "torus", 2 * SLABS + 5, 2, "start"), (256, "torus", 2 * SLABS + 5, 2, "dpsgd")])
def test_loads_that_stop_time_out_and_the_state_recovers(n, kind, d, K, mode):
    from test_gpu_failure_detection import _rebind
    m = _graph(kind, n)
    rng = np.random.default_rng(n)
    state = {k: rng.standard_normal((n, d), dtype=np.float32) for k in ("x", "y", "g", "a", "c")}
    got = []
    for stalled in (False, True):
        with Session(m, d, K, 0.2, 0.01, sigma=0.1, seed=5, gradient_point=int(mode == "start"), algorithm=int(mode == "dpsgd")) as s:
            if stalled:
                B.detag_debug_inject_stall(s.state, 1, 2048)
                s.step()
                with pytest.raises(B.DetagError) as e:
                    s.status()
                assert e.value.code == B.DETAG_ERR_TIMEOUT
                B.detag_debug_inject_stall(s.state, -1, 0)
                _rebind(s)
            for k, v in state.items():
                s.upload(k, v)
            B.detag_set_step(s.state, 0)
            s.step()
            s.status()
            assert B.detag_debug_kernel(s.state) == "step_split"
            got.append({k: s.download(k) for k in ("x", "y", "g")})
    assert all(np.array_equal(got[0][k], got[1][k]) for k in got[0])
