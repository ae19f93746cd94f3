"""What a launch mode makes of a domain's steps, read from a capture of them: programmatic or ordinary
edges between the kernels."""
import ctypes

import numpy as np
import pytest

import ttsh_inputs as ti

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    from paper_2304_03306_gb300 import build, ttsh
    build.build()
    ttsh.load_library()
    return ttsh


@pytest.fixture(scope="module")
def cu():
    lib = ctypes.CDLL("libcuda.so.1")
    P, S = ctypes.c_void_p, ctypes.POINTER(ctypes.c_size_t)
    lib.cuStreamBeginCapture_v2.argtypes = [P, ctypes.c_int]
    lib.cuStreamEndCapture.argtypes = [P, ctypes.POINTER(P)]
    lib.cuGraphGetEdges_v2.argtypes = [P, P, P, P, S]
    lib.cuGraphDestroy.argtypes = [P]
    lib.cuGraphGetNodes.argtypes = [P, P, S]
    lib.cuGraphKernelNodeGetParams_v2.argtypes = [P, P]
    return lib


def domain(T, n, prec):
    d = T.Domain(ti.circle_mask(n, 20.48 / n, 5.2), n, 20.48 / n, precision=prec)
    d.init_noise(3, 0.3)
    return d


def capture(cu, d, stream, steps):
    """Graph of the domain's next steps (the state does not move)."""
    d.set_stream(stream.cuda_stream)
    d.step(1)   # the kernels' attributes, before the capture
    d.synchronize()
    graph = ctypes.c_void_p()
    assert cu.cuStreamBeginCapture_v2(stream.cuda_stream, 1) == 0   # this thread's calls
    d.step(steps)
    assert cu.cuStreamEndCapture(stream.cuda_stream, ctypes.byref(graph)) == 0
    return graph


def programmatic_edges(cu, d, stream, steps=3):
    """(edges, programmatic edges) between the kernels of `steps` steps."""
    graph = capture(cu, d, stream, steps)
    k = ctypes.c_size_t(0)
    assert cu.cuGraphGetEdges_v2(graph, None, None, None, ctypes.byref(k)) == 0
    a, b = (ctypes.c_void_p * k.value)(), (ctypes.c_void_p * k.value)()
    data = (ctypes.c_ubyte * (8 * k.value))()   # CUgraphEdgeData: from_port, to_port, type, five reserved bytes
    assert cu.cuGraphGetEdges_v2(graph, a, b, data, ctypes.byref(k)) == 0
    cu.cuGraphDestroy(graph)
    return k.value, sum(data[8 * i + 2] == 1 for i in range(k.value))


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("n", [64, 1024])
def test_bit_0_decides_whether_passes_overlap(T, cu, n, prec):
    torch = pytest.importorskip("torch")
    stream = torch.cuda.Stream()
    d = domain(T, n, prec)
    for mode in (0, 1, 2, 3, 0):
        p = d.plan()
        d.set_plan(p["row_variant"], p["col_variant"], launch_mode=mode)
        edges, programmatic = programmatic_edges(cu, d, stream)
        assert edges == 5 and programmatic == (5 if mode & 1 else 0), mode
        assert d.plan()["launch_mode"] == mode
    d.synchronize()
    d.close()


@pytest.mark.parametrize("prec", [32, 64])
def test_autotuned_small_grid_reports_overlapped_launches(T, cu, prec):
    torch = pytest.importorskip("torch")
    stream = torch.cuda.Stream()
    d = domain(T, 64, prec)
    assert programmatic_edges(cu, d, stream)[1] == 5   # no mode set: overlapped on a small grid
    plan = d.autotune(iters=20)
    assert plan["launch_mode"] & 1
    assert programmatic_edges(cu, d, stream)[1] == 5
    d.synchronize()
    d.close()


@pytest.mark.parametrize("n,prec", [(64, 32), (512, 32), (1024, 32), (64, 64), (1024, 64)])
def test_overlapped_and_ordinary_launches_leave_the_same_bits(T, n, prec):
    """Graph replays, steps launched one by one and recorded steps, in every mode and in none."""
    def run(mode):
        d = domain(T, n, prec)
        if mode is not None:
            p = d.plan()
            d.set_plan(p["row_variant"], p["col_variant"], launch_mode=mode)
        d.step(270)   # graph replays and steps one by one
        series = d.record(150, 10)
        w, v = d.spectral_state()
        d.close()
        return w, v, series

    ref = run(0)
    for mode in (None, 1):
        got = run(mode)
        assert all(np.array_equal(x, y) for x, y in zip(ref, got)), mode


@pytest.mark.parametrize("prec", [32, 64])
def test_captured_steps_of_a_large_grid_are_ordinary_launches(T, cu, prec):
    """While no mode is set, steps beyond 512^2 overlap one by one and not in a graph, whoever
    records it (a corrected rollout's period, a caller)."""
    torch = pytest.importorskip("torch")
    stream = torch.cuda.Stream()
    d = domain(T, 1024, prec)
    assert programmatic_edges(cu, d, stream) == (5, 0)
    d.synchronize()
    d.close()


class KernelParams(ctypes.Structure):   # CUDA_KERNEL_NODE_PARAMS_v2
    _fields_ = [("func", ctypes.c_void_p), ("grid", ctypes.c_uint * 3), ("block", ctypes.c_uint * 3),
                ("shared", ctypes.c_uint), ("params", ctypes.c_void_p), ("extra", ctypes.c_void_p),
                ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("n", [16, 64, 128, 256, 512])
def test_a_step_leaves_room_on_an_sm_for_another_domain(T, cu, n, prec):
    """A pass of fewer blocks than SMs does not keep the blocks of domains on other streams off its
    SMs: two blocks fit (228 KB; 1 KB is the runtime's, up to 1 KB static)."""
    torch = pytest.importorskip("torch")
    stream = torch.cuda.Stream()
    d = domain(T, n, prec)
    graph = capture(cu, d, stream, 1)
    k = ctypes.c_size_t(0)
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(k)) == 0 and k.value == 2
    nodes = (ctypes.c_void_p * k.value)()
    assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(k)) == 0
    for node in nodes:
        q = KernelParams()
        assert cu.cuGraphKernelNodeGetParams_v2(node, ctypes.byref(q)) == 0
        if q.grid[0] <= 148:
            assert 2 * (q.shared + 2048) <= 228 * 1024, (list(q.grid), q.shared)
    cu.cuGraphDestroy(graph)
    d.synchronize()
    d.close()
