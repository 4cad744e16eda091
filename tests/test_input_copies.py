"""Inputs that a call copies first (not contiguous): the copy's stream and lifetime (needs a GB300)."""

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def busy(n=30):
    """Some milliseconds of work on the current stream."""
    a = torch.ones((4096, 4096), device="cuda")
    for _ in range(n):
        a = a @ a * 1e-4
    return a


def test_copy_for_another_stream():
    from paper_2110_01172_gb300 import Plan, PoissonSolver
    shape = (1024, 512)
    plan, solver, side = Plan(shape), PoissonSolver(shape), torch.cuda.Stream()
    xs = [torch.rand(shape, generator=torch.Generator(device="cuda").manual_seed(i), device="cuda") for i in range(6)]
    ref, ref_p = [plan.forward(x).clone() for x in xs], [solver.solve(x)[0].clone() for x in xs]
    ts = [x.t().contiguous().t() for x in xs]
    outs, fields = [torch.empty_like(x) for x in xs], [[torch.empty_like(x) for _ in range(3)] for x in xs]
    assert not ts[0].is_contiguous()
    torch.cuda.synchronize()
    for stream in (side, torch.cuda.ExternalStream(side.cuda_stream)):
        keep = busy()  # the copies queue up behind this
        for t, out, field in zip(ts, outs, fields):
            plan.forward(t, out, stream=stream)
            solver.solve(t, *field, stream=stream)
            torch.empty(shape, device="cuda").fill_(7)  # takes the copy's memory if it was given back too soon
        torch.cuda.synchronize()
        assert keep is not None
        assert all(torch.equal(o, r) for o, r in zip(outs, ref))
        assert all(torch.equal(f[0], r) for f, r in zip(fields, ref_p))
        [o.zero_() for o in outs]


@pytest.mark.parametrize("shape", [(64, 64), (1024, 2048), (64, 512)])
def test_page_locked_input_that_is_not_contiguous(shape):
    from paper_2110_01172_gb300 import Plan
    plan = Plan(shape)
    x = torch.rand(shape[::-1], generator=torch.Generator().manual_seed(3)).pin_memory().t()
    assert x.is_pinned() and not x.is_contiguous()
    ref = plan.forward(x.cuda().contiguous()).cpu()
    outs = [plan.forward(x) for _ in range(8)]
    torch.cuda.synchronize()
    for out in outs:
        assert out.is_pinned() and ((out - ref).norm() / ref.norm()).item() <= 1e-6


def test_contiguous_input_is_not_copied():
    from paper_2110_01172_gb300 import binding
    x = torch.rand((8, 8), device="cuda")
    assert binding._contiguous(x, torch.cuda.Stream(), x.device) is x
