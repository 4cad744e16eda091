"""Plans of one FFT length with few and with many sequences share kernels and do not
take each other's shared-memory limit (needs a GB300)."""

import pytest

import oracle
from paper_2110_01172_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wide,narrow", [((1024, 8), (1024, 2)), ((8, 2048), (2, 2048)), ((16384, 8), (16384, 2)),
                                         ((512, 8), (512, 4))])
def test_a_later_narrow_plan_leaves_the_wide_one_usable(wide, narrow):
    from paper_2110_01172_gb300 import Plan
    first, second = Plan(wide), Plan(narrow)
    for plan, shape in ((first, wide), (second, narrow), (first, wide)):
        x = inputs.uniform(shape, seed=6)
        X = plan.forward(torch.from_numpy(x).cuda())
        back = plan.inverse(X).cpu().double().numpy()
        got, ref = X.cpu().double().numpy(), oracle.dct2_2d(x)
        assert ((got - ref) ** 2).sum() <= (1e-5) ** 2 * (ref ** 2).sum()
        assert ((back - x) ** 2).sum() <= (2e-5) ** 2 * (x.astype(float) ** 2).sum()


def test_uneven_batch_of_every_small_shape():
    from paper_2110_01172_gb300 import MultiPlan
    shapes = [(2 << i, 2 << j) for i in range(10) for j in range(10)]
    xs = [torch.from_numpy(inputs.uniform(s, seed=i)) for i, s in enumerate(shapes)]
    for graph in (False, True):
        m = MultiPlan(shapes, graph=graph)
        X = m.forward(m.pack(xs))
        back = m.inverse(X)
        for x, y in zip(xs, m.unpack(back)):
            assert ((y.cpu() - x).norm() / x.norm()).item() <= 2e-5
        m.close()
