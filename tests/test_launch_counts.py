"""gbdct_plan_launches against the kernel nodes of a captured call, and the names
of a plan's launches (needs a GB300)."""

import ctypes

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def captured_nodes(call, x, out):
    """Nodes of the graph that `call` (stream -> None) records."""
    driver = ctypes.CDLL("libcuda.so.1")
    stream = torch.cuda.Stream()
    handle, graph, count = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p(), ctypes.c_size_t()
    torch.cuda.synchronize()
    assert driver.cuStreamBeginCapture_v2(handle, 1) == 0
    call(stream)
    assert driver.cuStreamEndCapture(handle, ctypes.byref(graph)) == 0
    assert driver.cuGraphGetNodes(graph, None, ctypes.byref(count)) == 0
    assert driver.cuGraphDestroy(graph) == 0
    return count.value


@pytest.mark.parametrize("shape,kind,batch,family,split", [
    ((256, 512), "dct2", 1, None, False),      # two-pass
    ((64, 64), "dct2", 3, None, False),        # one launch
    ((16, 32), "dst2", 1, None, False),        # map kernels around the core
    ((8192, 256), "dct2", 1, None, False),     # four-step
    ((16, 64, 64), "dct2", 1, None, False),    # slices and the axis-0 pass
    ((256, 256), "dct2", 1, None, True),       # split products
    ((128, 128), "dct2", 100, None, True),
])
def test_launches_of_a_call(shape, kind, batch, family, split):
    from paper_2110_01172_gb300 import Plan
    plan = Plan(shape, kind, batch=batch, family=family)
    if split:
        plan.set_precision("split_bf16")
    x = torch.rand(((batch,) if batch > 1 else ()) + shape, device="cuda")
    out = torch.empty_like(x)
    plan.forward(x, out), plan.inverse(x, out)
    for inverse in (False, True):
        run = plan.inverse if inverse else plan.forward
        count = captured_nodes(lambda s: run(x, out, stream=s), x, out)
        assert plan.launches(inverse) == count
        names = [plan.step_name(inverse, k) for k in range(count)]
        assert all(names) and plan.step_name(inverse, count) == ""
    assert plan.launches_per_exec == plan.launches(False)
