"""A tuned 3D plan is the same plan every time it is asked for, also where the
default plan of its slices runs kernels that no family name selects (needs a
GB300)."""

import pytest

import oracle
from paper_2110_01172_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(16, 64, 64), (32, 32, 64), (128, 128, 128), (16, 64, 512), (8, 256, 256)])
def test_tuned_volume_is_reused(shape):
    from paper_2110_01172_gb300 import Plan
    x = torch.rand(shape, generator=torch.Generator(device="cuda").manual_seed(2), device="cuda")
    first, again = Plan(shape, tuned=True), Plan(shape, tuned=True)
    assert first.choice == again.choice and first.launches_per_exec == again.launches_per_exec
    X = first.forward(x)
    assert torch.equal(X, again.forward(x)) and torch.equal(first.inverse(X), again.inverse(X))
    back = first.inverse(X)
    assert ((back - x).norm() / x.norm()).item() <= 1e-5


def test_tuned_choice_names_a_plan_that_can_be_asked_for():
    """`choice` stays a family name that Plan(family=...) takes."""
    from paper_2110_01172_gb300 import Plan
    for shape in ((64, 64), (64, 512), (512, 512)):
        choice = Plan(shape, tuned=True).choice
        x = inputs.uniform(shape, seed=3)
        got = Plan(shape, family=choice).forward(torch.from_numpy(x).cuda()).cpu().double().numpy()
        ref = oracle.dct2_2d(x)
        assert ((got - ref) ** 2).sum() <= (1e-5) ** 2 * (ref ** 2).sum()
