"""The dense product of 17 to 48 workers by groups of warps: worker counts on and off the quads and output blocks, vectors below,
at and beyond a slab of 64 and what all groups take at a time, ragged last slabs, all modes, one step against the oracle per
element; infinities reach the workers that hear of them and no others."""
import numpy as np
import pytest

from oracle import detag_oracle as orc
from paper_2006_08085_b200 import binding as B
from paper_2006_08085_b200 import build, inputs
from paper_2006_08085_b200.session import Session
from parity import HALF_ULP32, oracle_problem, worst_ratio

pytestmark = pytest.mark.gpu

ROUND = 64 * 148  # a slab per SM; a group of warps has three or four of them before it


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


@pytest.mark.parametrize("n", [17, 20, 23, 26, 32, 33, 37, 44, 48])
@pytest.mark.parametrize("d", [1, 30, 65, ROUND + 64, 9 * ROUND + 35])
@pytest.mark.parametrize("mode", ["new", "start", "external", "dpsgd"])
def test_one_step_against_the_oracle(n, d, mode):
    m = inputs.metropolis_weights(inputs.random_regular4_graph(n, n))
    rng = np.random.default_rng(n * 131 + d)
    a = rng.uniform(0.5, 2.0, (n, d)).astype(np.float32)
    c, x, y, g, g_new = (rng.standard_normal((n, d)).astype(np.float32) for _ in range(5))
    K, eta, alpha, ld = 2, 0.25, 0.03, (d + 3) // 4 * 4 + 4
    with Session(m, d, K, eta, alpha, sigma=0.1, seed=7, coord_offset=5, ld=ld, observe_gossip=mode != "dpsgd",
                 gradient_point=int(mode == "start"), external_gradient=mode == "external",
                 algorithm=int(mode == "dpsgd")) as s:
        for k, v in (("a", a), ("c", c), ("x", x), ("y", y), ("g", g)) + ((("g_new", g_new),) if mode == "external" else ()):
            s.upload(k, v)
        for t in (s.x, s.y, s.g):
            t[:, d:] = 7.0
        B.detag_set_step(s.state, 0)
        s.step()
        s.status()
        got = {k: s.download(k) for k in ("x", "y", "g")}
        seen = s.download("y_gossip") if mode != "dpsgd" else None
        for t in (s.x, s.y, s.g):
            assert bool((t[:, d:] == 7.0).all())  # nothing beyond column d
    # the oracle on the first and last columns, and on every 97th between them
    take = np.unique(np.concatenate([np.arange(min(d, 70)), np.arange(max(0, d - 70), d), np.arange(0, d, 97)]))
    for lo, hi in _runs(take):
        p = oracle_problem(m, K, eta, alpha, a[:, lo:hi], c[:, lo:hi], 0.1, 7, 5 + lo)
        x_, y_, g_ = (v[:, lo:hi].astype(np.float64) for v in (x, y, g))
        out = {k: v[:, lo:hi] for k, v in got.items()}
        if mode == "dpsgd":
            want = orc.dpsgd_step(p, orc.DpsgdState(x_, g_, 0))
            assert worst_ratio(out["x"], want.x) <= 1.0 and worst_ratio(out["g"], want.g) <= 1.0
            assert np.array_equal(out["y"], y_)
            continue
        folded = y_ + g_new[:, lo:hi] - g_ if mode == "external" else y_
        x_new, y_gossip = orc.gossip_and_update(p, x_, folded)
        assert worst_ratio(out["x"], x_new) <= 1.0 and worst_ratio(seen[:, lo:hi], y_gossip) <= 1.0
        if mode == "external":
            assert worst_ratio(out["y"], y_gossip) <= 1.0 and np.array_equal(out["g"], g_new[:, lo:hi])
            continue
        g_ref = orc.stochastic_gradient(p, x_ if mode == "start" else x_new, 1)
        assert worst_ratio(out["g"], g_ref) <= 1.0
        assert worst_ratio(out["y"], y_gossip + g_ref - g_, extra=HALF_ULP32 * np.abs(g_ref)) <= 1.0


@pytest.mark.parametrize("n", [20, 32, 41, 48])
@pytest.mark.parametrize("mode", ["new", "start", "external", "dpsgd"])
def test_a_shard_of_the_coordinates_gives_what_the_whole_gives(n, mode):
    """Bit for bit, at lengths below and beyond a slab per SM."""
    m = inputs.metropolis_weights(inputs.random_regular4_graph(n, n))
    d, cut = 2 * ROUND + 100, ROUND - 60
    rng = np.random.default_rng(n)
    arrays = {k: rng.standard_normal((n, d)).astype(np.float32) for k in ("x", "y", "g", "a", "c") + (("g_new",) if mode == "external" else ())}
    got = []
    for lo, hi in ((0, d), (0, cut), (cut, 2 * cut), (2 * cut, d)):
        with Session(m, hi - lo, 4, 0.2, 0.05, sigma=0.1, seed=3, coord_offset=lo, gradient_point=int(mode == "start"),
                     external_gradient=mode == "external", algorithm=int(mode == "dpsgd")) as s:
            for k, v in arrays.items():
                s.upload(k, v[:, lo:hi])
            B.detag_set_step(s.state, 0)
            s.step(3)
            s.status()
            got.append([s.download(k) for k in ("x", "y", "g")])
    for k in range(3):
        assert np.array_equal(got[0][k], np.concatenate([part[k] for part in got[1:]], axis=1))


@pytest.mark.parametrize("n,bad", [(33, np.inf), (40, np.nan), (48, -np.inf)])
@pytest.mark.parametrize("mode", ["new", "external", "dpsgd"])
def test_what_is_not_finite_reaches_those_that_hear_of_it(n, bad, mode):
    m = inputs.metropolis_weights(inputs.ring_graph(n))
    d, K, worker = 2 * ROUND + 9, 2, 5
    cols = (3, ROUND + 11, d - 1)
    rng = np.random.default_rng(n)
    arrays = {k: rng.standard_normal((n, d)).astype(np.float32) for k in ("x", "y", "g", "a", "c", "g_new")}
    for col in cols:
        arrays["x"][worker, col] = bad
    with Session(m, d, K, 0.2, 0.05, sigma=0.1, seed=3, external_gradient=mode == "external", algorithm=int(mode == "dpsgd")) as s:
        for k, v in arrays.items():
            if getattr(s, k) is not None:
                s.upload(k, v)
        B.detag_set_step(s.state, 0)
        s.step()
        s.status()
        got = s.download("x")
    hears = np.abs((np.arange(n) - worker + n // 2) % n - n // 2) <= K
    finite = np.isfinite(got)
    for col in cols:
        assert np.array_equal(finite[:, col], ~hears)
    assert finite[:, np.setdiff1d(np.arange(d), cols)].all()


@pytest.mark.parametrize("n,d", [(33, 61), (44, 64 * 444 + 61), (48, 3)])
@pytest.mark.parametrize("mode", ["new", "external", "dpsgd"])
def test_what_is_not_finite_in_a_ragged_slab(n, d, mode):
    """The first slab of its group and a later one; one worker's model is infinite in every column, and the workers that do not
    hear of it get what they get without it."""
    m = inputs.metropolis_weights(inputs.ring_graph(n))
    K, cols = 2, np.arange(d // 64 * 64, d)
    rng = np.random.default_rng(n + d)
    arrays = {k: rng.standard_normal((n, d)).astype(np.float32) for k in ("x", "y", "g", "a", "c", "g_new")}
    got = []
    for bad in (False, True):
        with Session(m, d, K, 0.2, 0.05, sigma=0.1, seed=3, external_gradient=mode == "external", algorithm=int(mode == "dpsgd")) as s:
            for k, v in arrays.items():
                if getattr(s, k) is not None:
                    s.upload(k, v)
            if bad:
                s.x[cols % n, cols] = float("inf")
            B.detag_set_step(s.state, 0)
            s.step()
            s.status()
            got.append(s.download("x")[:, cols])
    hears = np.abs((np.arange(n)[:, None] - cols[None, :] % n + n // 2) % n - n // 2) <= K
    assert np.array_equal(np.isfinite(got[1]), ~hears)
    assert worst_ratio(got[1][~hears], got[0][~hears].astype(np.float64)) <= 1.0


def _runs(cols):
    ends = np.flatnonzero(np.diff(cols) != 1)
    return [(int(cols[a]), int(cols[b]) + 1) for a, b in zip(np.r_[0, ends + 1], np.r_[ends, len(cols) - 1])]
