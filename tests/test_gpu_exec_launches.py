"""fftu_exec_launches against what fftu_exec puts on a stream: the kernel nodes of its capture into a CUDA graph, for plans of
whole-axis tile passes (programmatic launches), of two phases, and with the layout permutations; the graph, launched on other
data, gives what fftu_exec gives, beside work on another stream."""
import ctypes

import numpy as np
import pytest

from fftu_inputs import complex_uniform

pytestmark = pytest.mark.gpu

CASES = [((64, 64, 64), None, {}), ((1024, 1024), None, {}), ((32, 32, 32, 32, 32), None, {}), ((16,), None, {}), ((2, 8192), None, {}),
         ((64, 64, 64), (2, 2, 2), {}), ((32, 32, 32), (4, 4, 4), {"schedule": 1}), ((64, 64, 64), None, {"layout": 1}),
         ((128, 64, 512), (2, 2, 8), {}), ((1024, 64), (4, 4), {"layout": 1})]


def ok(rc):
    assert rc == 0, rc


@pytest.mark.parametrize("dt", [np.complex64, np.complex128])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c[0])) + ("" if c[1] is None else "p") +
                         "".join(f"{k}{v}" for k, v in c[2].items()))
def test_launches_of_one_exec(case, dt):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2203_11795_gb300 as fftu
    rt = ctypes.CDLL(f"libcudart.so.{torch.version.cuda.split('.')[0]}")
    shape, p, options = case
    x = torch.from_numpy(complex_uniform(970, shape, dtype=dt)).cuda()
    other = torch.from_numpy(complex_uniform(971, shape, dtype=dt)).cuda()
    side, y = torch.cuda.Stream(), torch.empty_like(x)
    with fftu.Plan(shape, p, dtype=x.dtype, **options) as plan:
        want, expect = plan.exec(other), fftu.fftu_exec_launches(plan.handle)
        torch.cuda.synchronize()
        s, graph, run, n = ctypes.c_void_p(side.cuda_stream), ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_size_t()
        ok(rt.cudaStreamBeginCapture(s, 1))
        plan.exec(x, y, stream=side)
        ok(rt.cudaStreamEndCapture(s, ctypes.byref(graph)))
        ok(rt.cudaGraphGetNodes(graph, None, ctypes.byref(n)))
        nodes = (ctypes.c_void_p * n.value)()
        ok(rt.cudaGraphGetNodes(graph, nodes, ctypes.byref(n)))
        kernels = 0
        for node in nodes:
            kind = ctypes.c_int()
            ok(rt.cudaGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)))
            kernels += kind.value == 0
        assert kernels == expect
        x.copy_(other)
        ok(rt.cudaGraphInstantiate(ctypes.byref(run), graph, ctypes.c_ulonglong(0)))
        busy = torch.empty(1 << 22, device="cuda")
        torch.cuda.synchronize()
        for _ in range(3):
            ok(rt.cudaGraphLaunch(run, s))
            busy.normal_()
        torch.cuda.synchronize()
        assert torch.equal(y, want)
        ok(rt.cudaGraphExecDestroy(run))
        ok(rt.cudaGraphDestroy(graph))


def test_server_counts_what_it_launches():
    """Solo requests of default-grid plans: kernel_launches is requests times fftu_exec_launches."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2203_11795_gb300 as fftu
    shape, count = (64, 32, 64), 3
    with fftu.Plan(shape, None) as plan:
        each = fftu.fftu_exec_launches(plan.handle)
    bufs = [(torch.from_numpy(complex_uniform(980 + i, shape, dtype=np.complex64)).pin_memory(),
             torch.empty(shape, dtype=torch.complex64).pin_memory()) for i in range(count)]
    s = fftu.fftu_server_create(large_elems=1024)
    try:
        for i, (x, y) in enumerate(bufs):
            fftu.fftu_server_submit(s, shape, fftu.FFTU_C64, fftu.FFTU_FORWARD, x.data_ptr(), y.data_ptr(), i)
        fftu.fftu_server_drain(s, 60.0)
        stats = fftu.fftu_server_stats_get(s)
    finally:
        fftu.fftu_server_destroy(s)
    assert stats["completed"] == count and stats["kernel_launches"] == count * each
