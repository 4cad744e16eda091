"""Forward transforms of two-pass plans into page-locked host buffers, at the row
lengths whose output rows the row pass gathers before it stores them (needs a GB300)."""

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(64, 512), (64, 8192), (512, 64), (8192, 64), (512, 128), (128, 1024), (128, 4096),
                                   (64, 1024), (64, 2048), (128, 512), (8192, 128), (128, 256)])
@pytest.mark.parametrize("kind", ["dct2", "dst2"])
def test_host_output_equals_device_output(shape, kind):
    from paper_2110_01172_gb300 import Plan
    for batch in (1, 5):
        full = ((batch,) if batch > 1 else ()) + shape
        plan = Plan(shape, kind, batch=batch)
        x = torch.rand(full, generator=torch.Generator(device="cuda").manual_seed(4), device="cuda").sub_(0.5)
        ref = plan.forward(x).cpu()
        for source in (x, x.cpu().pin_memory()):
            out = torch.full(full, float("nan"), pin_memory=True)
            plan.forward(source, out)
            torch.cuda.synchronize()
            assert torch.equal(out, ref)
        if plan.family == "tp":  # the threshold goes with either store
            eps = float(ref.abs().median())
            plan.set_threshold(eps)
            out = torch.full(full, float("nan"), pin_memory=True)
            plan.forward(x, out)
            torch.cuda.synchronize()
            assert torch.equal(out, torch.where(ref.abs() < eps, torch.zeros_like(ref), ref))
        plan.close()


@pytest.mark.parametrize("shape", [(512, 64), (2048, 64), (512, 128)])
def test_host_output_is_no_slower_than_the_inverses(shape):
    """Both directions write the same bytes over the host link; stores of a few columns
    at a time made the forward two to four times as long."""
    from paper_2110_01172_gb300 import Plan
    plan = Plan(shape, batch=16)
    x = torch.rand((16,) + shape, device="cuda")
    out = torch.empty((16,) + shape, pin_memory=True)
    best = {}
    for run in (plan.forward, plan.inverse):
        for _ in range(12):
            start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            start.record()
            for _ in range(10):
                run(x, out)
            end.record()
            torch.cuda.synchronize()
            best[run.__name__] = min(best.get(run.__name__, 1e9), start.elapsed_time(end) * 100)
    print(shape, best)
    assert best["forward"] <= 1.5 * best["inverse"]
