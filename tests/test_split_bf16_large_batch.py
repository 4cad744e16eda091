"""Split-BF16 mode over more tile rows than a grid's y axis holds (65535): the
second product stacks the batch's rows of N2, so sides with N2 > N1 reach that
number first (needs a GB300)."""

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BOUND = 5e-5  # the mode's bound in relative L2, as for single transforms


def rel(got, ref):
    d = torch.stack([(g.double() - r.double()).square().sum() for g, r in zip(got, ref)]).sqrt()
    return (d / torch.stack([r.double().square().sum() for r in ref]).sqrt()).max().item()


def test_more_than_65535_tile_rows():
    from paper_2110_01172_gb300 import Plan
    batch, n1, n2 = 4096, 128, 2048
    assert batch * n2 // 128 > 65535
    gen = torch.Generator(device="cuda").manual_seed(7)
    x = torch.rand((batch, n1, n2), generator=gen, device="cuda").mul_(2).sub_(1)
    some = torch.tensor([0, 1, batch // 2 - 1, batch - 2, batch - 1], device="cuda")
    plan = Plan((n1, n2), batch=batch)
    X = plan.forward(x)[some]
    plan.set_precision("split_bf16")
    S = plan.forward(x)
    assert rel(S[some], X) <= BOUND
    y = plan.inverse(S)
    assert rel(y[some], x[some]) <= 2 * BOUND  # both directions' errors
    assert rel(y[::64], x[::64]) <= 2 * BOUND
    assert plan.check_device_error() == 0
    plan.close()
