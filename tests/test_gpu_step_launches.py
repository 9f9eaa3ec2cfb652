"""Runs under a caller's stream capture: qw_plan_step_launches counts the kernel nodes of a captured run, and replaying
a captured run or evolution (overlapped launches become programmatic edges) gives the fields of the plain calls."""

import ctypes

import pytest

from paper_1603_06442_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def qb(qwlib):
    from paper_1603_06442_gb300 import binding
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return binding


def field(dim, N, dtype):
    g = torch.Generator(device="cuda").manual_seed(N)
    return torch.randn(inputs.field_shape(dim, N), dtype=torch.complex64 if dtype == "c64" else torch.complex128,
                       device="cuda", generator=g)


def kernel_nodes(call, stream):
    """Kernel nodes of the graph that the call's capture on the stream gives (the driver's own count)."""
    cuda = ctypes.CDLL("libcuda.so.1")

    def ok(status):
        assert status == 0, status

    graph, n = ctypes.c_void_p(), ctypes.c_size_t()
    ok(cuda.cuStreamBeginCapture_v2(ctypes.c_void_p(stream.cuda_stream), 1))  # thread local
    try:
        call()
    finally:
        ok(cuda.cuStreamEndCapture(ctypes.c_void_p(stream.cuda_stream), ctypes.byref(graph)))
    ok(cuda.cuGraphGetNodes(graph, None, ctypes.byref(n)))
    nodes = (ctypes.c_void_p * n.value)()
    ok(cuda.cuGraphGetNodes(graph, nodes, ctypes.byref(n)))
    kernels = 0
    for node in nodes:
        kind = ctypes.c_int()
        ok(cuda.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)))
        kernels += kind.value == 0
    ok(cuda.cuGraphDestroy(graph))
    return kernels


@pytest.mark.parametrize("dim,N,dtype,variant", [
    (1, 1000, "c64", "auto"), (1, 1000, "c128", "auto"), (1, 4_000_000, "c128", "auto"), (2, 300, "c64", "auto"),
    (2, 300, "c128", "auto"), (3, 128, "c64", "auto"), (3, 512, "c64", "auto"), (3, 48, "c128", "auto"),
    (3, 128, "c64", "tma2"), (3, 128, "c64", "vec"), (3, 40, "c64", "fused"), (2, 64, "c64", "fused")])
@pytest.mark.parametrize("t", [1, 7, 100])
def test_launches_of_a_run(qb, dim, N, dtype, variant, t):
    plan = qb.Plan(dim, N, 0.2, dtype)
    plan.set_stencil(variant)
    x = field(dim, N, dtype)
    plan.step(x, t)
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    assert plan.step_launches(t) == kernel_nodes(lambda: plan.step(x, t, stream), stream)
    assert plan.step_launches(0) == 0 and plan.step_launches(-1) == -1
    plan.close()


@pytest.mark.parametrize("dim,N,dtype", [(1, 1024, "c64"), (1, 1024, "c128"), (2, 300, "c64"), (3, 48, "c128"),
                                         (3, 128, "c64"), (3, 384, "c64")])
@pytest.mark.parametrize("t", [1, 2, 9])
def test_a_captured_run_replays(qb, dim, N, dtype, t):
    plan = qb.Plan(dim, N, 0.2, dtype)
    x, want = field(dim, N, dtype), field(dim, N, dtype)
    for _ in range(4):
        plan.step(want, t)
    plan.step(x, t)  # as many steps before the capture as it will replay after
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        plan.step(x, t)
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    plan.sync()
    plan.close()
    assert torch.equal(x, want)


@pytest.mark.parametrize("dim,N,dtype", [(1, 1024, "c128"), (1, 1 << 16, "c64"), (2, 64, "c128"), (3, 32, "c64")])
def test_a_captured_evolution_replays(qb, dim, N, dtype):
    plan = qb.Plan(dim, N, 0.2, dtype)
    x, want = field(dim, N, dtype), field(dim, N, dtype)
    fw_want = None
    for _ in range(4):
        plan.evolve_spectral(want, 7)
        fw_want = plan.fw_transform(want)
    plan.evolve_spectral(x, 7)
    fw = torch.empty_like(x)
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        plan.evolve_spectral(x, 7)
        plan.fw_transform(x, out=fw)
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    plan.close()
    assert torch.equal(x, want) and torch.equal(fw, fw_want)
