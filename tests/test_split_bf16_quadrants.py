"""The split-BF16 mode's half-size products at the edges of its shapes: sides whose
quadrants are smaller than a tile, uneven sides, odd batches, in place, against
the oracle.

Error allowed: each operand is within 2^-17 of its hi + lo parts (relative to its
magnitude), four roundings enter a result (two products, two operands each), and
the round trip has twice as many: 4 * 2^-17 = 3.1e-5 in the worst case of equal
signs, half of that (1.5e-5) where they are independent.
"""

import numpy as np
import pytest

import oracle
from paper_2110_01172_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,batch", [((128, 128), 1), ((128, 128), 3), ((128, 2048), 1), ((2048, 128), 1),
                                         ((256, 128), 5), ((128, 512), 2), ((1024, 256), 3)])
def test_quadrants(shape, batch):
    from paper_2110_01172_gb300 import Plan, binding
    xs = np.stack([inputs.uniform(shape, seed=80 + i) for i in range(batch)])
    x = torch.from_numpy(xs if batch > 1 else xs[0]).cuda()
    plan = Plan(shape, batch=batch).set_precision("split_bf16")
    X, y = plan.forward(x), plan.inverse(x)
    for run, out in ((plan.forward, X), (plan.inverse, y)):
        z = x.clone()
        run(z, out=z)
        assert torch.equal(z, out)
    for i in range(batch):
        for got, ref in ((X, oracle.dct2_2d(xs[i])), (y, oracle.idct2_2d(xs[i]))):
            got = (got[i] if batch > 1 else got).cpu().numpy().astype(np.float64)
            assert np.linalg.norm(got - ref) <= 1.5e-5 * np.linalg.norm(ref)
    assert plan.check_device_error() == binding.OK
    plan.close()
