"""The circulant band kernel (K * bandwidth <= 16) over several slabs per block: reuse of the ring of chunks, of the side copy
and of the stages from slab to slab, both gradient points, D-PSGD, and the columns beyond the last whole slab."""
import numpy as np
import pytest

from oracle import detag_oracle as orc
from paper_2006_08085_b200 import binding as B
from paper_2006_08085_b200 import build, inputs
from paper_2006_08085_b200.session import Session
from parity import HALF_ULP32, oracle_problem, worst_ratio

pytestmark = pytest.mark.gpu

SLABS = 64 * 148  # one slab of 64 coordinates per block


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def _matrix(kind, n):
    if kind == "ring":
        return inputs.metropolis_weights(inputs.ring_graph(n))
    return inputs.directed_cycle_blend(n, 0.4, 0.35)


@pytest.mark.parametrize("n,d,K,kind", [
    (64, 3 * SLABS + 5, 16, "ring"), (96, 2 * SLABS + 65, 1, "directed"), (256, 3 * SLABS + 7, 4, "ring"),
    (288, 3 * SLABS + 5, 5, "directed"), (512, 2 * SLABS + 130, 16, "ring"), (1024, SLABS + 64, 3, "ring")])
@pytest.mark.parametrize("mode", ["new", "start", "dpsgd"])
def test_one_step_against_the_oracle(n, d, K, kind, mode):
    m = _matrix(kind, n)
    eta, alpha = 0.3, 0.02
    rng = np.random.default_rng(n + d)
    a = rng.random((n, d), dtype=np.float32) + np.float32(0.5)
    c, x0, y0, g0 = (rng.standard_normal((n, d), dtype=np.float32) for _ in range(4))
    with Session(m, d, K, eta, alpha, a, c, x0, 0.1, 11, observe_gossip=mode != "dpsgd", variant=B.DETAG_VARIANT_RING,
                 gradient_point=int(mode == "start"), algorithm=int(mode == "dpsgd")) as s:
        s.upload("y", y0)
        s.upload("g", g0)
        B.detag_set_step(s.state, 0)
        s.step()
        s.status()
        got = {k: s.download(k) for k in ("x", "y", "g") + (() if mode == "dpsgd" else ("y_gossip",))}
    w = m.to_dense()
    prev = P = np.eye(n)
    for _ in range(K):
        prev, P = P, (1.0 + eta) * w @ P - eta * prev
    # a few stretches of columns: both ends, and one in every slab of the first and of the last block
    starts = {0, 30, d - 70, *(64 * (148 * k) + 20 for k in range(d // SLABS + 1)),
              *(64 * (148 * k + 147) + 10 for k in range(d // SLABS + 1))}
    for lo in sorted(v for v in starts if v < d):
        cut = slice(lo, min(d, lo + 70))
        x, y, g = (v[:, cut].astype(np.float64) for v in (x0, y0, g0))
        p = oracle_problem(m, K, eta, alpha, a[:, cut], c[:, cut], 0.1, 11, lo)
        y_gossip = P @ y
        x_new = P @ x - alpha * (g if mode == "dpsgd" else y_gossip)
        g_new = orc.stochastic_gradient(p, x if mode == "start" else x_new, 1)
        assert worst_ratio(got["x"][:, cut], x_new) <= 1.0, (lo, "x")
        assert worst_ratio(got["g"][:, cut], g_new) <= 1.0, (lo, "g")
        if mode == "dpsgd":
            assert np.array_equal(got["y"][:, cut], y0[:, cut])
            continue
        assert worst_ratio(got["y_gossip"][:, cut], y_gossip) <= 1.0, (lo, "y_gossip")
        assert worst_ratio(got["y"][:, cut], y_gossip + g_new - g, extra=HALF_ULP32 * np.abs(g_new)) <= 1.0, (lo, "y")


@pytest.mark.parametrize("n,worker,K,bad", [(64, 63, 16, np.inf), (96, 0, 3, np.nan), (256, 31, 1, -np.inf), (288, 270, 5, np.inf)])
def test_what_is_not_finite_stays_in_reach(n, worker, K, bad):
    """One operand of the model and one of the tracker; the band's zeros must not carry them further, also around the end."""
    d, eta = 128, 0.2
    m = _matrix("ring", n)
    x, y = np.random.default_rng(n).standard_normal((2, n, d)).astype(np.float32)
    x[worker, 9] = bad
    y[worker, 64] = bad
    zero = np.zeros((n, d), np.float32)
    with Session(m, d, K, eta, 0.0, zero, zero, x, observe_gossip=True, variant=B.DETAG_VARIANT_RING) as s:
        s.upload("y", y)
        B.detag_set_step(s.state, 0)
        s.step()
        s.status()
        got = {"x": s.download("x"), "y_gossip": s.download("y_gossip")}
    P = np.eye(n)
    prev, w = P, m.to_dense()
    for _ in range(K):
        prev, P = P, (1.0 + eta) * w @ P - eta * prev
    reached = P[:, worker] != 0.0
    assert reached.sum() == 2 * K + 1
    for (name, z), col in zip((("x", x), ("y_gossip", y)), (9, 64)):
        assert not np.isfinite(got[name][reached, col]).any(), name
        keep = np.ones((n, d), bool)
        keep[reached, col] = False
        if name == "x":
            keep[reached, 64] = False  # x' = P x - 0 * P y
        z[worker, col] = 0.0
        assert worst_ratio(got[name][keep], (P @ z.astype(np.float64))[keep]) <= 1.0, name


@pytest.mark.parametrize("n,d,K", [(128, 64 * 200 + 3, 4), (160, 65, 3), (192, 64 * 150 + 33, 16), (256, 3001, 2), (288, 1000, 5)])
def test_ragged_steps_in_a_row_give_the_bits_of_steps_one_by_one(n, d, K):
    """The columns beyond the last whole slab are a launch of their own that runs beside the band's."""
    m = inputs.metropolis_weights(inputs.ring_graph(n))
    rng = np.random.default_rng(n)
    state = {k: rng.standard_normal((n, d)).astype(np.float32) for k in ("x", "y", "g", "a", "c")}
    got = []
    for together in (False, True):
        with Session(m, d, K, 0.2, 0.01, sigma=0.1, seed=9) as s:
            for k, v in state.items():
                s.upload(k, v)
            for _ in range(12):
                s.step()
                if not together:
                    s.torch.cuda.synchronize()
            s.status()
            got.append({k: s.download(k) for k in ("x", "y", "g")})
    assert all(np.array_equal(got[0][k], got[1][k]) for k in got[0])


@pytest.mark.parametrize("n,d,K,mode", [(64, 3 * 64 + 5, 16, "new"), (64, SLABS - 3, 4, "start"), (96, 2 * SLABS + 64, 14, "new"), (128, SLABS + 33, 16, "dpsgd"),
                                        (160, 131, 16, "new")])
def test_the_variant_chosen_by_name_runs_in_float64_throughout(n, d, K, mode):
    """Every sum is a float64 one rounded once, whatever the width of the band and the length: also where the sum cancels to a
    hundred-thousandth of what it reads, of which fixed point of 39 bits would leave an error of 2^-21."""
    m, eta = _matrix("ring", n), 0.2
    prev, w = np.eye(n), m.to_dense()
    P = prev
    for _ in range(K):
        prev, P = P, (1.0 + eta) * w @ P - eta * prev
    x, y = np.random.default_rng(n + d).standard_normal((2, n, d)).astype(np.float32)
    zero = np.zeros((n, d), np.float32)
    with Session(m, d, K, eta, 0.0, zero, zero, x, observe_gossip=mode != "dpsgd", variant=B.DETAG_VARIANT_RING, gradient_point=int(mode == "start"),
                 algorithm=int(mode == "dpsgd")) as s:
        s.upload("y", y)
        s.step()
        s.status()
        got = {"x": (s.download("x"), x)}
        if mode != "dpsgd":
            got["y"] = (s.download("y_gossip"), y)
        ran = [B.detag_debug_kernel(s.state, part) for part in (0, 1)]
    assert ran == ["step_ring", "step_csr" if d % 64 != 0 else ""]
    for name, (have, z) in got.items():
        want, reads = P @ z.astype(np.float64), np.abs(P) @ np.abs(z.astype(np.float64))
        bound = 2.0 ** -24 * np.abs(want) + 2.0 ** -46 * reads + 1e-45
        assert (np.abs(have - want) <= bound).all(), name


@pytest.mark.parametrize("n,d,K,algorithm,ran", [
    (64, 60_032, 12, 0, ("step_ring", "")), (96, 200_001, 16, 0, ("step_ring", "step_rows")), (128, 60_001, 16, 0, ("step_ring", "step_rows")),
    (128, 4096, 16, 1, ("step_ring", "")), (256, 3_001, 4, 0, ("step_ring", "step_csr")), (64, 4 * 32 * 148 + 1, 4, 0, ("step_ring", "step_rows")),
    (64, 3_001, 4, 0, ("step_rows", "")), (128, 3_001, 16, 0, ("step_rows", "")), (128, 32 * 148 + 1, 4, 1, ("step_ring", "step_rows"))])
def test_bands_stay_in_float64_but_for_the_last_columns_and_short_ragged_calls(n, d, K, algorithm, ran):
    with Session(_matrix("ring", n), d, K, 0.2, 0.01, algorithm=algorithm) as s:
        s.step()
        s.status()
        assert tuple(B.detag_debug_kernel(s.state, part) for part in (0, 1)) == ran
