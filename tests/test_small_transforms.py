"""Small transforms in one launch (one CTA each): every shape it is built for,
every kind, batches that leave part of the last CTA idle, buffers in place,
against the oracle; what such plans accept and refuse."""

import numpy as np
import pytest

import oracle
from paper_2110_01172_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

REL_L2, MAX_ABS = 1e-5, 1e-4  # the tolerance of every FP32 result against the oracle
SHAPES = [(1 << a, 1 << b) for a in range(5, 10) for b in range(5, 10) if a + b <= 14]
KINDS = {"dct2": (oracle.dct2_2d, oracle.idct2_2d), "dst2": (oracle.dst2_2d, oracle.idst2_2d),
         "idct_idxst": (None, oracle.idct_idxst), "idxst_idct": (None, oracle.idxst_idct)}


def check(got, ref):
    got, ref = got.cpu().numpy().astype(np.float64), np.asarray(ref, np.float64)
    assert np.linalg.norm(got - ref) <= REL_L2 * np.linalg.norm(ref)
    assert np.abs(got - ref).max() <= MAX_ABS * np.abs(ref).max()


@pytest.mark.parametrize("kind", list(KINDS))
@pytest.mark.parametrize("shape", SHAPES)
def test_every_shape_and_kind(shape, kind):
    from paper_2110_01172_gb300 import Plan
    fwd, inv = KINDS[kind]
    # 128 x 128 takes this path for batches only
    for batch in (1, 3) if shape != (128, 128) else (160, 161):
        xs = np.stack([inputs.uniform(shape, seed=50 + i) for i in range(batch)])
        x = torch.from_numpy(xs if batch > 1 else xs[0]).cuda()
        plan = Plan(shape, kind, batch=batch)
        assert plan.launches_per_exec == 1 and plan.step_name(False, 0)
        for ref, run in ((fwd, plan.forward), (inv, plan.inverse)):
            if ref is None:
                continue
            y = run(x)
            z = x.clone()
            run(z, out=z)
            assert torch.equal(y, z)
            for i in range(batch) if batch < 8 else (0, 77, batch - 1):
                check(y[i] if batch > 1 else y, ref(xs[i]))
        plan.close()


def test_threshold_and_host_buffers_as_before():
    from paper_2110_01172_gb300 import GbdctError, Plan
    x = torch.from_numpy(np.stack([inputs.uniform((128, 128), seed=9 + i) for i in range(160)]))
    plan = Plan((128, 128), batch=160)
    assert plan.launches_per_exec == 1
    X = plan.forward(x.cuda())
    eps = float(X.abs().median())
    plan.set_threshold(eps)
    assert torch.equal(plan.forward(x.cuda()), torch.where(X.abs() < eps, torch.zeros_like(X), X))
    plan.set_threshold(0.0)
    host = plan.forward(x.pin_memory())
    torch.cuda.synchronize()
    assert torch.equal(host, X.cpu())
    with pytest.raises(GbdctError):
        Plan((64, 128)).set_threshold(eps)
    assert Plan((128, 128)).launches_per_exec == 2 and Plan((128, 128), batch=200).launches_per_exec == 1
    assert Plan((64, 64)).family == "pair" and Plan((64, 64), family="pair").launches_per_exec == 2


def test_tuned_plan_is_reused():
    from paper_2110_01172_gb300 import Plan
    x = torch.from_numpy(inputs.uniform((64, 64), seed=9)).cuda()
    first, again = Plan((64, 64), tuned=True), Plan((64, 64), tuned=True)
    assert first.choice == again.choice and first.launches_per_exec == again.launches_per_exec
    check(again.forward(x), oracle.dct2_2d(x.cpu().numpy()))
