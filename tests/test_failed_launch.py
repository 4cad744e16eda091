"""A launch that fails is reported by its own call and by no later one (needs a GB300)."""

import ctypes

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,split", [((256, 512), False), ((8192, 256), False), ((64, 64), False), ((256, 256), True)])
def test_the_next_plan_is_created(shape, split):
    """The launch fails on the host: its stream's capture has been given up before it."""
    from paper_2110_01172_gb300 import GbdctError, Plan
    driver = ctypes.CDLL("libcuda.so.1")
    plan = Plan(shape)
    if split:
        plan.set_precision("split_bf16")
    x = torch.rand(shape, device="cuda")
    out = torch.empty_like(x)
    ref = plan.forward(x).clone()
    stream = torch.cuda.Stream()
    handle, graph = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p()
    torch.cuda.synchronize()
    assert driver.cuStreamBeginCapture_v2(handle, 1) == 0
    assert driver.cuStreamSynchronize(handle) != 0  # not permitted in a capture, which it ends as invalid
    with pytest.raises(GbdctError):
        plan.forward(x, out, stream=stream)
    assert driver.cuStreamEndCapture(handle, ctypes.byref(graph)) != 0
    assert torch.equal(Plan(shape).forward(x), ref if not split else Plan(shape).forward(x))
    assert torch.equal(plan.forward(x), ref)
