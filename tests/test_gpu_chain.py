"""Steps that follow one another on a stream, each launch beginning while the one before it finishes: the same bits as with the
device idle between them, on every kernel, from a captured graph too, and between other work on the stream."""
import numpy as np
import pytest

from paper_2006_08085_b200 import binding as B
from paper_2006_08085_b200 import build, inputs
from paper_2006_08085_b200.session import Session

pytestmark = pytest.mark.gpu

CASES = [  # n, d, K, graph, variant, mode
    (8, 4096, 2, "ring", B.DETAG_VARIANT_AUTO, "detag"), (16, 33_001, 2, "ring", B.DETAG_VARIANT_AUTO, "external"),
    (24, 20_003, 3, "regular4", B.DETAG_VARIANT_AUTO, "detag"), (30, 20_003, 3, "regular4", B.DETAG_VARIANT_AUTO, "external"),
    (48, 30_001, 3, "regular4", B.DETAG_VARIANT_AUTO, "detag"), (64, 20_010, 4, "torus", B.DETAG_VARIANT_AUTO, "detag"),
    (100, 30_002, 4, "regular4", B.DETAG_VARIANT_AUTO, "detag"), (256, 3_003, 9, "torus", B.DETAG_VARIANT_AUTO, "detag"),
    (96, 40_005, 4, "ring", B.DETAG_VARIANT_AUTO, "detag"),  # band kernel, its last columns in a launch of their own
    (60, 5_003, 3, "regular4", B.DETAG_VARIANT_CSR, "detag"),
    (90, 20_003, 4, "regular4", B.DETAG_VARIANT_AUTO, "detag"), (60, 160_010, 4, "regular4", B.DETAG_VARIANT_AUTO, "detag"),  # step_split
    (256, 6_003, 2, "torus", B.DETAG_VARIANT_AUTO, "dpsgd"), (160, 6_002, 2, "torus", B.DETAG_VARIANT_AUTO, "detag"),
    (144, 20_003, 8, "regular4", B.DETAG_VARIANT_AUTO, "detag"), (100, 20_003, 6, "regular4", B.DETAG_VARIANT_AUTO, "external"),  # step_rows
    (160, 20_003, 40, "ring", B.DETAG_VARIANT_AUTO, "external"),
    (256, 20_005, 4, "ring", B.DETAG_VARIANT_AUTO, "detag"), (96, 20_005, 9, "ring", B.DETAG_VARIANT_RING, "dpsgd")]  # band, rounds beside it

KERNELS = {(8, "ring"): "step_small", (16, "ring"): "step_small", (24, "regular4"): "step_dense", (30, "regular4"): "step_mma", (48, "regular4"): "step_dense",
           (64, "torus"): "step_torus", (96, "ring"): "step_ring", (90, "regular4"): "step_split", (256, "torus"): ("step_rows", "step_split"),
           (160, "torus"): "step_split", (144, "regular4"): "step_rows", (100, "regular4"): "step_rows", (160, "ring"): "step_rows", (256, "ring"): "step_ring"}


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def _session(n, d, K, graph, variant, mode):
    m = inputs.metropolis_weights(inputs.ring_graph(n) if graph == "ring" else inputs.torus_graph(n // 8, 8)
                                  if graph == "torus" else inputs.random_regular4_graph(n, n))
    rng = np.random.default_rng(n + d)
    s = Session(m, d, K, 0.2, 0.02, sigma=0.1, seed=5, variant=variant, external_gradient=mode == "external",
                algorithm=B.DETAG_ALGORITHM_DPSGD if mode == "dpsgd" else B.DETAG_ALGORITHM_DETAG)
    for k in ("x", "y", "g", "a", "c") + (("g_new",) if mode == "external" else ()):
        s.upload(k, rng.standard_normal((n, d)).astype(np.float32))
    B.detag_set_step(s.state, 0)
    return s


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"{c[0]}-{c[3]}-{c[5]}-{c[1]}")
def test_back_to_back_as_with_the_device_idle_between(case):
    import torch

    got = []
    for how in ("idle", "chained", "captured"):
        with _session(*case) as s:
            stream = torch.cuda.Stream()
            stream.wait_stream(torch.cuda.current_stream())

            def steps(count):
                for _ in range(count):
                    if s.g_new is not None:  # another kernel between the steps, which the next one reads from
                        s.g_new.mul_(0.5)
                    s.step()
                    if how == "idle":
                        torch.cuda.synchronize()

            with torch.cuda.stream(stream):
                steps(2)
                if how == "captured":
                    stream.synchronize()
                    graph, t = torch.cuda.CUDAGraph(), B.detag_get_step(s.state)
                    with torch.cuda.graph(graph, stream=stream):
                        steps(6)
                    assert B.detag_get_step(s.state) == t + 6
                    graph.replay()
                else:
                    steps(6)
            stream.synchronize()
            s.status()
            assert B.detag_debug_kernel(s.state) in KERNELS.get(case[::3][:2], ("step_split", "step_csr"))  # 60 workers: by length, by name
            got.append({k: s.download(k) for k in ("x", "y", "g")})
    for other in got[1:]:
        for k in ("x", "y", "g"):
            assert np.array_equal(got[0][k], other[k]), k


@pytest.mark.parametrize("n", [8, 24, 60])
def test_a_launch_that_fails_is_reported_once(n):
    """A step on a stream whose capture was broken off fails at its launch; the next call knows nothing of it."""
    import ctypes

    import torch

    cu = ctypes.CDLL("libcuda.so.1")
    with _session(n, 4096, 2, "ring", B.DETAG_VARIANT_AUTO, "detag") as s:
        s.step()
        torch.cuda.synchronize()
        handle = ctypes.c_void_p(torch.cuda.Stream().cuda_stream)
        assert cu.cuStreamBeginCapture_v2(handle, 1) == 0   # thread-local
        assert cu.cuStreamSynchronize(handle) != 0          # not allowed there: ends the capture
        with pytest.raises(B.DetagError) as e:
            B.detag_step(s.state, handle.value)
        assert e.value.code == B.DETAG_ERR_CUDA
        graph = ctypes.c_void_p()
        assert cu.cuStreamEndCapture(handle, ctypes.byref(graph)) != 0
        B.detag_init(s.state, handle.value)
        B.detag_step(s.state, handle.value)
        s.consensus_error()
        torch.cuda.synchronize()
        s.status()
