"""Default plans with a side of 64 (too large for one launch) run the two-pass
kernels: every kind, batches, in place and host buffers against the oracle, and
what such plans are called, accept and refuse."""

import numpy as np
import pytest

import oracle
from paper_2110_01172_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

REL_L2, MAX_ABS = 1e-5, 1e-4  # the tolerance of every FP32 result against the oracle
KINDS = {"dct2": (oracle.dct2_2d, oracle.idct2_2d), "dst2": (oracle.dst2_2d, oracle.idst2_2d),
         "idct_idxst": (None, oracle.idct_idxst), "idxst_idct": (None, oracle.idxst_idct)}


def check(got, ref):
    got, ref = got.cpu().numpy().astype(np.float64), np.asarray(ref, np.float64)
    assert np.linalg.norm(got - ref) <= REL_L2 * np.linalg.norm(ref)
    assert np.abs(got - ref).max() <= MAX_ABS * np.abs(ref).max()


@pytest.mark.parametrize("kind", list(KINDS))
@pytest.mark.parametrize("shape,batch", [((64, 512), 1), ((512, 64), 1), ((64, 1024), 3), ((1024, 64), 5),
                                         ((64, 8192), 1), ((8192, 64), 1), ((2048, 64), 2), ((64, 512), 41)])
def test_every_kind(shape, batch, kind):
    from paper_2110_01172_gb300 import Plan
    fwd, inv = KINDS[kind]
    xs = np.stack([inputs.uniform(shape, seed=60 + i) for i in range(batch)])
    x = torch.from_numpy(xs if batch > 1 else xs[0]).cuda()
    plan = Plan(shape, kind, batch=batch)
    assert plan.launches_per_exec == 2 and plan.step_name(False, 1)
    for ref, run in ((fwd, plan.forward), (inv, plan.inverse)):
        if ref is None:
            continue
        y = run(x)
        z = x.clone()
        run(z, out=z)
        assert torch.equal(y, z)
        host = run(x.cpu().pin_memory())
        torch.cuda.synchronize()
        for i in {0, batch - 1}:
            check(y[i] if batch > 1 else y, ref(xs[i]))
            check(host[i] if batch > 1 else host, ref(xs[i]))
    assert plan.check_device_error() == 0
    plan.close()


def test_names_and_refusals_as_before():
    from paper_2110_01172_gb300 import GbdctError, Plan
    plan = Plan((64, 512))
    assert plan.family == "pair"
    with pytest.raises(GbdctError):
        plan.set_threshold(0.5)
    with pytest.raises(GbdctError):
        Plan((64, 512), family="tp")
    x = torch.from_numpy(inputs.uniform((64, 512), seed=3)).cuda()
    first, again = Plan((64, 512), tuned=True), Plan((64, 512), tuned=True)
    assert first.choice == again.choice and torch.equal(first.forward(x), again.forward(x))
    forced = Plan((64, 512), "dst2", family="pair")
    assert forced.family == "pair" and forced.launches_per_exec == 4
