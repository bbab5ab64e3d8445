"""The integer tensor path with output workers as lanes (step_rows.cu): the sizes at which its plan changes (64, 128 workers, planes of
the polynomial in tensor memory or through a ring), caller-written gradients, coordinates summed in float64."""
import numpy as np
import pytest

from paper_2006_08085_b200 import build, inputs
from paper_2006_08085_b200.session import Session
from test_gpu_split import (_graph, _polynomial, _unequal, patterns_side_by_side, test_dpsgd as dpsgd, test_every_result_is_as_precise_as_what_it_reads as precision,
                            test_one_step_against_the_oracle as one_step, test_what_is_not_finite_stays_in_reach as not_finite)

pytestmark = pytest.mark.gpu

CHUNKS = 32 * 148  # one chunk of 32 coordinates per block


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


@pytest.fixture
def kernels(monkeypatch):
    """Names of the kernels that the steps before every status() ran on."""
    from paper_2006_08085_b200 import binding as B
    seen, plain = set(), Session.status

    def status(self):
        seen.add(B.detag_debug_kernel(self.state))
        plain(self)

    monkeypatch.setattr(Session, "status", status)
    return seen


# below, at and beyond a chunk, one and several per block and (beyond 16 per block) chunks in pairs; odd numbers of chunks
@pytest.mark.parametrize("n,d,K,kind,at_start", [
    (49, 31, 3, "regular4", False), (64, 33, 4, "ring", True), (64, 17 * CHUNKS + 33, 3, "regular4", False), (65, 3 * CHUNKS + 5, 3, "path", False),
    (97, 17 * CHUNKS + 2, 4, "regular4", True), (128, 18 * CHUNKS + 31, 5, "regular4", False),
    (129, 65, 4, "ring", False), (130, 3 * CHUNKS + 5, 6, "path", False), (150, 5 * CHUNKS + 67, 2, "regular4", True), (161, 130, 7, "directed", False),
    (200, 63, 12, "regular4", False), (255, 2 * CHUNKS + 3, 9, "ring", True), (256, 17 * CHUNKS + 66, 5, "regular4", False)])
def test_one_step(n, d, K, kind, at_start):
    one_step(n, d, K, kind, at_start)


# ... of them those whose dispatch chooses other kernels, at numbers of rounds and lengths where it chooses this one
@pytest.mark.parametrize("n,d,K,kind,at_start", [
    (65, 3 * CHUNKS // 4, 3, "path", False), (96, 31, 9, "regular4", True), (130, 31, 20, "regular4", False), (161, 130, 24, "regular4", True), (200, 63, 20, "regular4", False),
    (256, 1, 20, "regular4", True), (181, 150, 40, "ring", False), (160, 33, 40, "ring", True), (256, CHUNKS + 66, 9, "torus", False)])
def test_one_step_of_this_kernel(n, d, K, kind, at_start, kernels):
    one_step(n, d, K, kind, at_start)
    assert kernels == {"step_rows"}


@pytest.mark.parametrize("kind,n,K", [("regular4", 144, 16), ("ring", 181, 60), ("regular4", 256, 16), ("ring", 192, 40)])
def test_precision_of_this_kernel_beyond_128_workers(kind, n, K, kernels):
    precision(kind, n, K)
    assert kernels == {"step_rows"}


# from one to all of eight coordinates of either array in float64, or of both; chunks with and without them in turn
@pytest.mark.parametrize("n,kind,d,K,mode", [(60, "regular4", 2_003, 2, "detag"), (50, "path", 3 * CHUNKS + 1, 6, "dpsgd"), (80, "regular4", 3_001, 2, "start"),
                                             (70, "ring", 1_999, 4, "dpsgd"), (100, "path", 2 * CHUNKS + 3, 3, "detag"), (128, "regular4", 18 * CHUNKS + 1, 6, "start"),
                                             (112, "regular4", 2_001, 1, "dpsgd"), (144, "regular4", 2_003, 16, "detag"), (160, "ring", 4_003, 20, "start"),
                                             (256, "regular4", 3 * CHUNKS, 12, "detag"), (256, "torus", 2 * CHUNKS + 1, 9, "dpsgd")])
def test_float64_columns_beside_split_ones(n, kind, d, K, mode):
    patterns_side_by_side(n, kind, d, K, mode, "step_rows")


@pytest.mark.parametrize("n,d,K", [(144, 130, 16), (171, 131, 24), (256, 5 * CHUNKS + 9, 12)])
@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_dpsgd_and_what_is_not_finite_beyond_128_workers(n, d, K, bad, kernels):
    """D-PSGD, and DeTAG's tracker: dense polynomials, so what is not finite reaches everyone - in its own column and array."""
    from paper_2006_08085_b200 import binding as B
    m, eta, alpha = _graph("regular4", n), 0.2, 0.05
    P = _polynomial(m, K, eta)
    rng = np.random.default_rng(n)
    x, y, g = (rng.standard_normal((n, d), dtype=np.float32) for _ in range(3))
    x[9, 40] = bad
    y[n - 1, 70] = bad
    zero = np.zeros((n, d), np.float32)
    cols = np.unique(np.concatenate([np.arange(130), np.arange(d - 100, d)]))
    fine = x[:, cols].astype(np.float64), y[:, cols].astype(np.float64), g[:, cols].astype(np.float64)
    for algorithm in (B.DETAG_ALGORITHM_DPSGD, B.DETAG_ALGORITHM_DETAG):
        with Session(m, d, K, eta, alpha, zero, zero, x, algorithm=algorithm, observe_gossip=algorithm == B.DETAG_ALGORITHM_DETAG) as s:
            s.upload("y", y)
            s.upload("g", g)
            s.step()
            s.status()
            got = s.download("x")[:, cols]
            yt = s.download("y_gossip")[:, cols] if algorithm == B.DETAG_ALGORITHM_DETAG else None
        with np.errstate(invalid="ignore"):
            want = P @ fine[0] - alpha * (fine[2] if yt is None else P @ fine[1])
        at = np.isin(cols, [40, 70] if yt is not None else [40])
        assert not np.isfinite(got[:, at]).any()
        assert (np.abs(got[:, ~at] - want[:, ~at]) <= 1e-5 * (1.0 + np.abs(want[:, ~at]))).all()
        if yt is not None:
            at = cols == 70
            assert not np.isfinite(yt[:, at]).any()
            with np.errstate(invalid="ignore"):
                want = P @ fine[1]
            assert (np.abs(yt[:, ~at] - want[:, ~at]) <= 1e-5 * (1.0 + np.abs(want[:, ~at]))).all()
    assert kernels == {"step_rows"}


@pytest.mark.parametrize("kind,n", [("regular4", 144), ("ring", 181), ("regular4", 256)])
@pytest.mark.parametrize("K", [3, 16])
def test_precision_beyond_128_workers(kind, n, K):
    precision(kind, n, K)


def test_dpsgd_and_infinities_beyond_128_workers():
    dpsgd(171, 5 * CHUNKS + 9)
    not_finite(171, np.inf)


@pytest.mark.parametrize("n,d,K,kind", [(49, 1, 1, "regular4"), (50, 35, 2, "ring"), (64, 2 * CHUNKS + 34, 4, "regular4"), (65, 97, 6, "path"),
                                        (100, 5 * CHUNKS + 7, 2, "regular4"), (128, 17 * CHUNKS + 33, 9, "regular4"), (129, 3 * CHUNKS + 35, 7, "path"),
                                        (160, 2 * CHUNKS + 1, 40, "ring"), (192, 4 * CHUNKS + 33, 6, "regular4"), (193, 65, 6, "regular4")])
def test_caller_written_gradients(n, d, K, kind):
    """x' = P x - alpha y', y' = P (y + g_new - g), g' = g_new: two steps, the second with operands of unequal size.  Bound: half an
    ulp of what is stored, and as much again relative to the magnitudes that the result reads for the sums; the folded operand itself
    carries 2^-40 of its three parts."""
    eta, alpha = 0.2, 0.05
    m = _graph(kind, n)
    P = _polynomial(m, K, eta)
    rng = np.random.default_rng(n + d)
    zero = np.zeros((n, d), np.float32)
    cols = slice(0, d) if d <= 5000 else np.unique(np.concatenate([np.arange(200), np.arange(d - 200, d), rng.integers(0, d, 400)]))
    with Session(m, d, K, eta, alpha, zero, zero, zero, external_gradient=True, observe_gossip=True) as s:
        for pattern in ("alike", "log-uniform"):
            state = {"x": _unequal(pattern, n, d, rng), "y": _unequal(pattern, n, d, rng), "g": (30 * rng.standard_normal((n, d))).astype(np.float32),
                     "g_new": (30 * rng.standard_normal((n, d))).astype(np.float32)}
            for k, v in state.items():
                s.upload(k, v)
            s.step()
            s.status()
            got = {k: s.download(k)[:, cols].astype(np.float64) for k in ("x", "y", "g", "y_gossip")}
            x, y, g, gn = (state[k][:, cols].astype(np.float64) for k in ("x", "y", "g", "g_new"))
            z, parts = y + gn - g, np.abs(y) + np.abs(gn) + np.abs(g)
            yt = P @ z
            of_y = 2.0 ** -24 * (np.abs(yt) + np.abs(P) @ np.abs(z)) + 2.0 ** -40 * (np.abs(P) @ parts) + 1e-45
            xt = P @ x - alpha * yt
            of_x = 2.0 ** -24 * (np.abs(xt) + np.abs(P) @ np.abs(x)) + alpha * of_y + 1e-45
            assert (np.abs(got["y"] - yt) <= of_y).all()
            assert (np.abs(got["x"] - xt) <= of_x).all()
            assert np.array_equal(got["g"], gn) and np.array_equal(got["y_gossip"], got["y"])


@pytest.mark.parametrize("n,kind", [(60, "regular4"), (90, "regular4"), (128, "regular4"), (160, "ring"), (192, "regular4")])
@pytest.mark.parametrize("K", [1, 2, 6, 16])
def test_caller_written_gradients_whose_fold_cancels(n, kind, K, kernels):
    """y + g_new - g far below its parts: the first step after detag_init (y = g) where gradients have fallen.  The bound knows the sum z
    alone: half an ulp of what is stored and as much again of the magnitudes read, nothing of the three parts (of which float64 itself
    loses 2^-53, here some 2^-28 of the sum)."""
    d, eta, alpha = 3 * CHUNKS + 35, 0.2, 0.05
    m = _graph(kind, n)
    P = _polynomial(m, K, eta)
    rng = np.random.default_rng(n + K)
    cols = np.unique(np.concatenate([np.arange(140), np.arange(d - 140, d), rng.integers(0, d, 500)]))
    f = np.float32
    x, y, g, gn = (rng.standard_normal((n, d), dtype=f) for _ in range(4))
    y[:] = g
    kind_of = np.arange(d) % 14
    for k in range(9):  # gradients that fall by 2^0, 2^-3, .. 2^-24
        gn[:, kind_of == k] *= f(2.0 ** (-3 * k))
    outlier = np.ix_([n // 3], np.flatnonzero(kind_of == 9))  # one worker's gradient was large, the others are what they were
    g[outlier] *= f(1e6)
    y[outlier] = g[outlier]
    at = kind_of == 10  # the float32 sum is zero at every worker, the exact one is not
    y[:, at] = g[:, at] = f(1.0) + rng.random((n, at.sum()), dtype=f)
    gn[:, at] = np.copysign(f(2.0 ** -25) * (f(1.0) + rng.random((n, at.sum()), dtype=f)), gn[:, at])
    at = kind_of == 11  # all but cancels
    y[:, at] *= f(1.0) + f(2.0 ** -20) * rng.standard_normal((n, at.sum()), dtype=f)
    gn[:, at] *= f(2.0 ** -14)
    at = kind_of == 12  # the gradients cancel, the tracker is small
    gn[:, at] = g[:, at] * (f(1.0) + f(2.0 ** -18) * rng.standard_normal((n, at.sum()), dtype=f))
    y[:, at] = f(2.0 ** -20) * rng.standard_normal((n, at.sum()), dtype=f)
    at = kind_of == 13  # the tracker cancels the new gradient
    y[:, at] = -gn[:, at]
    g[:, at] *= f(2.0 ** -24)
    zero = np.zeros((n, d), f)
    with Session(m, d, K, eta, alpha, zero, zero, zero, external_gradient=True) as s:
        for k, v in (("x", x), ("y", y), ("g", g), ("g_new", gn)):
            s.upload(k, v)
        s.step()
        s.status()
        got = {k: s.download(k)[:, cols].astype(np.float64) for k in ("x", "y", "g")}
    wide = np.longdouble
    z = (y[:, cols].astype(wide) - g[:, cols].astype(wide) + gn[:, cols].astype(wide)).astype(np.float64)
    x = x[:, cols].astype(np.float64)
    yt = P @ z
    of_y = 2.0 ** -24 * (np.abs(yt) + np.abs(P) @ np.abs(z)) + 1e-45
    xt = P @ x - alpha * yt
    of_x = 2.0 ** -24 * (np.abs(xt) + np.abs(P) @ np.abs(x)) + alpha * of_y + 1e-45
    worst = [float((np.abs(got["y"] - yt) / of_y)[:, cols % 14 == k].max()) for k in range(14)]
    assert max(worst) <= 1.0, [round(v, 2) for v in worst]
    assert (np.abs(got["x"] - xt) <= of_x).all()
    assert np.array_equal(got["g"], gn[:, cols])
    assert K < 16 or kernels == {"step_rows"}  # fewer rounds run as such, some of them


# one worker beyond a block, whole blocks, one beyond the first half; below, at and beyond a chunk
@pytest.mark.parametrize("n,d,K,kind", [(49, 1, 16, "regular4"), (50, 35, 30, "ring"), (64, 33, 12, "regular4"), (70, 97, 30, "ring"), (96, 31, 12, "regular4"),
                                        (97, CHUNKS + 34, 12, "regular4"), (129, 35, 14, "regular4"), (160, 3 * CHUNKS + 2, 16, "regular4"), (192, 31, 16, "regular4")])
def test_caller_written_gradients_of_this_kernel(n, d, K, kind, kernels):
    test_caller_written_gradients(n, d, K, kind)
    assert kernels == {"step_rows"}


@pytest.mark.parametrize("n,K", [(70, 30), (56, 30), (160, 40)])
def test_caller_written_gradients_of_this_kernel_that_are_not_finite(n, K, kernels):
    test_caller_written_gradients_that_are_not_finite(n, K)
    assert kernels == {"step_rows"}


def test_caller_written_gradients_that_are_not_finite(n=70, K=2):
    d, eta = 40, 0.2
    m = _graph("ring", n)
    P = _polynomial(m, K, eta)
    rng = np.random.default_rng(7)
    zero = np.zeros((n, d), np.float32)
    y, g, gn = (rng.standard_normal((n, d)).astype(np.float32) for _ in range(3))
    gn[9, 35] = np.inf
    with Session(m, d, K, eta, 0.0, zero, zero, zero, external_gradient=True) as s:
        for k, v in (("y", y), ("g", g), ("g_new", gn)):
            s.upload(k, v)
        s.step()
        s.status()
        got, g_out = s.download("y"), s.download("g")
    reached = P[:, 9] != 0.0
    assert not np.isfinite(got[reached, 35]).any()
    keep = np.ones((n, d), bool)
    keep[reached, 35] = False
    gn0 = np.where(np.isfinite(gn), gn, 0.0).astype(np.float64)
    want = P @ (y.astype(np.float64) + gn0 - g)
    assert (np.abs(got - want)[keep] <= 1e-5 * (1.0 + np.abs(want[keep]))).all()
    assert np.array_equal(g_out, gn)


@pytest.mark.parametrize("n,mode", [(60, "detag"), (90, "dpsgd"), (100, "detag"), (144, "detag"), (100, "external")])
def test_rows_further_apart_give_the_same_bits(n, mode):
    from paper_2006_08085_b200 import binding as B
    d, m = 3 * CHUNKS + 3, _graph("regular4", n)
    rng = np.random.default_rng(n)
    state = {k: rng.standard_normal((n, d)).astype(np.float32) for k in ("x", "y", "g", "a", "c", "g_new")}
    got = []
    for ld in (None, (d + 3) // 4 * 4 + 20):
        with Session(m, d, 6, 0.2, 0.01, sigma=0.1, seed=5, ld=ld, external_gradient=mode == "external",
                     algorithm=B.DETAG_ALGORITHM_DPSGD if mode == "dpsgd" else B.DETAG_ALGORITHM_DETAG) as s:
            for k, v in state.items():
                if k != "g_new" or mode == "external":
                    s.upload(k, v)
            s.step(2)
            s.status()
            got.append({k: s.download(k) for k in ("x", "y", "g")})
    assert all(np.array_equal(got[0][k], got[1][k]) for k in got[0])


@pytest.mark.parametrize("n,mode,after", [(60, "detag", 0), (60, "detag", 3), (90, "dpsgd", 2), (100, "detag", 1), (100, "external", 2), (144, "detag", 1),
                                          (144, "detag", 4), (150, "external", 2)])
def test_loads_that_stop_time_out_and_the_state_recovers(n, mode, after):
    """Some of a block's chunks are loaded, the others are not: every wait gives up and the launch ends; after re-binding the state steps
    to the bits of one that was never disturbed."""
    from paper_2006_08085_b200 import binding as B
    from test_gpu_failure_detection import _rebind
    d, m = 4 * CHUNKS + 5, _graph("regular4", n)
    rng = np.random.default_rng(n + after)
    state = {k: rng.standard_normal((n, d)).astype(np.float32) for k in ("x", "y", "g", "a", "c", "g_new")}
    got = []
    for stalled in (False, True):
        with Session(m, d, 6, 0.2, 0.01, sigma=0.1, seed=5, external_gradient=mode == "external",
                     algorithm=B.DETAG_ALGORITHM_DPSGD if mode == "dpsgd" else B.DETAG_ALGORITHM_DETAG) as s:
            if stalled:
                B.detag_debug_inject_stall(s.state, after, 2048)
                s.step()
                with pytest.raises(B.DetagError) as e:
                    s.status()
                assert e.value.code == B.DETAG_ERR_TIMEOUT
                B.detag_debug_inject_stall(s.state, -1, 0)
                _rebind(s)
            for k, v in state.items():
                if k != "g_new" or mode == "external":
                    s.upload(k, v)
            B.detag_set_step(s.state, 0)
            s.step()
            s.status()
            got.append({k: s.download(k) for k in ("x", "y", "g")})
    assert all(np.array_equal(got[0][k], got[1][k]) for k in got[0])


@pytest.mark.parametrize("n,mode", [(144, "detag"), (200, "start"), (256, "dpsgd")])
def test_the_gradient_beyond_128_workers_is_the_rounds(n, mode):
    """Matrices without block structure: a o (x' - c) + sigma xi in float64, rounded once, as on the rounds kernel.  The models differ by the
    fixed point's 1e-11 before they are rounded, which tips a few gradients in 10^5; a float32 product sigma xi tips one in five."""
    from paper_2006_08085_b200 import binding as B
    d, K, m = 5 * CHUNKS + 7, 12, _graph("regular4", n)
    rng = np.random.default_rng(n)
    state = {k: rng.standard_normal((n, d), dtype=np.float32) for k in ("x", "y", "g", "a", "c")}
    got = []
    for variant in (B.DETAG_VARIANT_AUTO, B.DETAG_VARIANT_CSR):
        with Session(m, d, K, 0.2, 0.01, sigma=0.3, seed=5, variant=variant, gradient_point=int(mode == "start"),
                     algorithm=int(mode == "dpsgd")) as s:
            for k, v in state.items():
                s.upload(k, v)
            s.step()
            s.status()
            got.append((s.download("g"), B.detag_debug_kernel(s.state)))
    assert [name for _, name in got] == ["step_rows", "step_csr"]
    assert np.count_nonzero(got[0][0] != got[1][0]) <= 2e-4 * n * d


@pytest.mark.parametrize("n,d,K,kind,mode,ran", [
    (100, 1_000_000, 2, "regular4", "external", "step_csr"), (100, 100_000, 4, "regular4", "external", "step_csr"), (100, 100_000, 6, "regular4", "external", "step_rows"),
    (144, 500_000, 3, "regular4", "external", "step_csr"), (160, 100_000, 16, "ring", "external", "step_rows"), (192, 100_000, 6, "regular4", "external", "step_rows"),
    (144, 400_000, 4, "regular4", "detag", "step_csr"), (215, 143_473, 6, "regular4", "detag", "step_rows"), (144, 100_000, 8, "regular4", "detag", "step_rows"), (256, 200_000, 4, "regular4", "detag", "step_csr"), (256, 200_000, 6, "regular4", "detag", "step_rows"),
    (256, 200_000, 3, "regular4", "dpsgd", "step_csr"), (256, 100_000, 12, "regular4", "detag", "step_rows")])
def test_few_rounds_on_sparse_graphs_stay_rounds(n, d, K, kind, mode, ran):
    """Operands that differ by four decades would send most coordinates of these to float64 on the integer path, at two to three times the
    rounds' time (100 workers, K = 2, caller-written gradients, d = 1 M: 5380 us against 1638)."""
    from paper_2006_08085_b200 import binding as B
    with Session(_graph(kind, n), d, K, 0.2, 0.01, external_gradient=mode == "external",
                 algorithm=B.DETAG_ALGORITHM_DPSGD if mode == "dpsgd" else B.DETAG_ALGORITHM_DETAG) as s:
        s.step()
        s.status()
        assert B.detag_debug_kernel(s.state) == ran
