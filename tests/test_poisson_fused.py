"""The fused Poisson solve (two-pass kernels over the three inverses at once)
against the oracle, at the edges of the shapes it takes and in the forms of
buffers and streams that a solve accepts."""

import numpy as np
import pytest

import oracle
from paper_2110_01172_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

REL_L2, MAX_ABS = 1e-5, 1e-4  # the tolerance of every FP32 result against the oracle


def check(outputs, rho):
    for got, ref in zip(outputs, oracle.poisson_solve(rho)):
        got, ref = got.cpu().numpy().astype(np.float64), np.asarray(ref, np.float64)
        assert np.linalg.norm(got - ref) <= REL_L2 * np.linalg.norm(ref)
        assert np.abs(got - ref).max() <= MAX_ABS * np.abs(ref).max()


@pytest.mark.parametrize("shape", [(64, 64), (64, 128), (128, 64), (64, 2048), (2048, 64), (64, 8192), (8192, 64),
                                   (128, 1024), (512, 512), (1024, 256), (4096, 128), (32, 64), (8192, 256)])
def test_shapes(shape):
    from paper_2110_01172_gb300 import PoissonSolver
    rho = inputs.density_blobs(shape, seed=3, n_blobs=40)
    solver = PoissonSolver(shape)
    check(solver.solve(torch.from_numpy(rho).cuda()), rho)
    solver.close()


@pytest.mark.parametrize("shape", [(64, 256), (256, 512)])
def test_buffers_streams_and_capture(shape):
    from paper_2110_01172_gb300 import PoissonSolver
    rho = inputs.density_blobs(shape, seed=4, n_blobs=40)
    solver = PoissonSolver(shape)
    x = torch.from_numpy(rho).cuda()
    plain = [t.clone() for t in solver.solve(x)]
    check(plain, rho)
    # the density's own buffer as an output
    for i in range(3):
        out = [torch.empty_like(x) for _ in range(3)]
        out[i] = x.clone()
        assert all(torch.equal(a, b) for a, b in zip(solver.solve(out[i], *out), plain))
    # captured and replayed on another stream
    out, g = [torch.zeros_like(x) for _ in range(3)], torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        solver.solve(x, *out)
    g.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(out, plain))
    # page-locked host outputs, through the C entry
    host = [torch.empty(shape, dtype=torch.float32, pin_memory=True) for _ in range(3)]
    assert solver._lib.gbdct_poisson_solve(solver._h, x.data_ptr(), *[t.data_ptr() for t in host], None) == 0
    torch.cuda.synchronize()
    check(host, rho)
    assert solver._lib.gbdct_poisson_solve(solver._h, x.data_ptr() + 4, *[t.data_ptr() for t in out], None) == 1
    solver.close()
