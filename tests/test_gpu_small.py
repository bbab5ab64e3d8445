"""At most 16 workers, the step in registers: worker counts on and off the quads, vectors below, at and beyond a block of
every size the launch picks (32, 64, 128 threads), all modes, one step against the oracle per element."""
import numpy as np
import pytest

from oracle import detag_oracle as orc
from paper_2006_08085_b200 import binding as B
from paper_2006_08085_b200 import build, inputs
from paper_2006_08085_b200.session import Session
from parity import HALF_ULP32, oracle_problem, worst_ratio

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


@pytest.mark.parametrize("n", [3, 4, 5, 8, 11, 12, 13, 16])
@pytest.mark.parametrize("d", [1, 33, 64 * 148 - 1, 64 * 148 + 65, 128 * 148 + 129])
@pytest.mark.parametrize("mode", ["new", "start", "external", "dpsgd"])
def test_one_step_against_the_oracle(n, d, mode):
    m = inputs.metropolis_weights(inputs.ring_graph(n))
    rng = np.random.default_rng(n * 131 + d)
    a = rng.uniform(0.5, 2.0, (n, d)).astype(np.float32)
    c, x, y, g, g_new = (rng.standard_normal((n, d)).astype(np.float32) for _ in range(5))
    K, eta, alpha = 3, 0.25, 0.03
    p = oracle_problem(m, K, eta, alpha, a, c, 0.1, 7, 5)
    with Session(m, d, K, eta, alpha, a, c, x, 0.1, 7, coord_offset=5, observe_gossip=mode != "dpsgd",
                 gradient_point=int(mode == "start"), external_gradient=mode == "external",
                 algorithm=int(mode == "dpsgd")) as s:
        s.upload("y", y)
        s.upload("g", g)
        if mode == "external":
            s.upload("g_new", g_new)
        B.detag_set_step(s.state, 0)
        s.step()
        s.status()
        got = {k: s.download(k) for k in ("x", "y", "g")}
        seen = s.download("y_gossip") if mode != "dpsgd" else None
    x, y, g = (v.astype(np.float64) for v in (x, y, g))
    if mode == "dpsgd":
        want = orc.dpsgd_step(p, orc.DpsgdState(x, g, 0))
        assert worst_ratio(got["x"], want.x) <= 1.0 and worst_ratio(got["g"], want.g) <= 1.0
        assert np.array_equal(got["y"], y)
        return
    folded = y + g_new - g if mode == "external" else y
    x_new, y_gossip = orc.gossip_and_update(p, x, folded)
    assert worst_ratio(got["x"], x_new) <= 1.0 and worst_ratio(seen, y_gossip) <= 1.0
    if mode == "external":
        assert worst_ratio(got["y"], y_gossip) <= 1.0 and np.array_equal(got["g"], g_new)
        return
    g_ref = orc.stochastic_gradient(p, x if mode == "start" else x_new, 1)
    assert worst_ratio(got["g"], g_ref) <= 1.0
    assert worst_ratio(got["y"], y_gossip + g_ref - g, extra=HALF_ULP32 * np.abs(g_ref)) <= 1.0


@pytest.mark.parametrize("n", [2, 6, 16])
@pytest.mark.parametrize("d", [2, 31, 32, 2 * 32 * 148 + 1, 4 * 32 * 148 + 3])
@pytest.mark.parametrize("steps", [1, 3])
def test_columns_keep_to_themselves(n, d, steps):
    """A warp's 16 or 32 coordinates, the vectors of a row and the blocks of the launch end anywhere: nothing beyond column d
    changes, and an infinity stays in its coordinate."""
    m = inputs.csr_from_dense(np.full((2, 2), 0.5)) if n == 2 else inputs.metropolis_weights(inputs.ring_graph(n))
    rng = np.random.default_rng(n * 17 + d)
    arrays = {k: rng.standard_normal((n, d)).astype(np.float32) for k in ("x", "y", "g", "a", "c")}
    hit = d // 2
    got = []
    for bad in (False, True):
        with Session(m, d, 2, 0.2, 0.05, sigma=0.1, seed=3, ld=(d + 3) // 4 * 4 + 4) as s:
            for k, v in arrays.items():
                s.upload(k, v)
                getattr(s, k)[:, d:] = 7.0
            if bad:
                s.x[0, hit] = float("inf")
            B.detag_set_step(s.state, 0)
            s.step_many(steps)
            s.status()
            got.append({k: getattr(s, k).cpu().numpy() for k in ("x", "y", "g")})
    keep = np.arange(d) != hit
    for k in ("x", "y", "g"):
        assert np.all(got[0][k][:, d:] == 7.0) and np.all(got[1][k][:, d:] == 7.0)
        assert np.all(np.isfinite(got[0][k])) and np.array_equal(got[0][k][:, :d][:, keep], got[1][k][:, :d][:, keep])
    assert not np.isfinite(got[1]["x"][0, hit])
