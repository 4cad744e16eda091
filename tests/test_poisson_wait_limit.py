"""A Poisson solve whose bounded waits give up says so, and the next one is right again
(needs a GB300; the limit of one poll makes the waits run out, nothing faults)."""

import ctypes

import pytest

import oracle
from paper_2110_01172_gb300 import binding, build, inputs

torch = pytest.importorskip("torch")


def test_null_solver():
    build.build()
    lib = binding.load()
    assert lib.gbdct_poisson_check_device_error(None) == binding.ERR_INVALID_ARG
    assert lib.gbdct_poisson_set_wait_limit(ctypes.c_void_p(), 1) == binding.ERR_INVALID_ARG


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(256, 512), (64, 64), (1024, 4096), (16, 64)])  # the last one: separate plans
def test_timeout_is_reported_and_recovers(shape):
    from paper_2110_01172_gb300 import PoissonSolver
    rho = inputs.density_blobs(shape, seed=8, n_blobs=40)
    x = torch.from_numpy(rho).cuda()
    solver = PoissonSolver(shape)
    solver.solve(x)
    assert solver.check_device_error() == binding.OK
    solver.set_wait_limit(1)
    solver.solve(x)
    torch.cuda.synchronize()
    waits = min(shape) >= 64  # the two-sequence kernels of a side of 16 wait for nothing
    assert solver.check_device_error() == (binding.ERR_TIMEOUT if waits else binding.OK)
    assert solver.check_device_error() == binding.OK
    solver.set_wait_limit(0)
    out = solver.solve(x)
    torch.cuda.synchronize()
    assert solver.check_device_error() == binding.OK
    for got, ref in zip(out, oracle.poisson_solve(rho)):
        got = got.cpu().double().numpy()
        assert ((got - ref) ** 2).sum() <= (1e-5) ** 2 * (ref ** 2).sum()
