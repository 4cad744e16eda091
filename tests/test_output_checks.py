"""Output tensors that the kernels would write past are refused before any launch
(needs a GB300)."""

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def bad_outputs(n):
    yield torch.empty(n - 4, device="cuda")
    yield torch.empty(n, device="cuda", dtype=torch.float16)
    yield torch.empty(2 * n, device="cuda")[::2]
    yield torch.empty(n)  # pageable


def test_refused_and_accepted():
    from paper_2110_01172_gb300 import MultiPlan, PoissonSolver
    from paper_2110_01172_gb300.binding import dct2_noalloc
    shape = (64, 128)
    n = shape[0] * shape[1]
    multi, solver = MultiPlan([shape, shape], graph=False), PoissonSolver(shape)
    x, rho = torch.rand(multi.total, device="cuda"), torch.rand(shape, device="cuda")
    for out in bad_outputs(multi.total):
        with pytest.raises(ValueError):
            multi.forward(x, out)
    for out in bad_outputs(n):
        with pytest.raises(ValueError):
            dct2_noalloc(rho, out)
        for i in range(3):
            with pytest.raises(ValueError):
                solver.solve(rho, **{("psi", "xi0", "xi1")[i]: out})
    ref = multi.forward(x)
    assert torch.equal(multi.forward(x, torch.empty(2, multi.total // 2, device="cuda")).reshape(-1), ref)
    fields = solver.solve(rho)
    flat = [torch.empty(n, device="cuda") for _ in range(3)]
    solver.solve(rho, *flat)
    assert all(torch.equal(f.view(shape), g) for f, g in zip(flat, fields))
    pinned = [torch.empty(shape, pin_memory=True) for _ in range(3)]
    solver.solve(rho, *pinned)
    torch.cuda.synchronize()
    assert all(((f - g.cpu()).norm() / f.norm()).item() <= 1e-5 for f, g in zip(pinned, fields))
