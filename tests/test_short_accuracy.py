"""Default plans with a side below 128 are as exact as the two-sequence kernels that
these shapes once ran, measured against 64 bits on the same inputs (needs a GB300).

The margin of 1.01 is the statistics of the comparison: with 2^20 values and more per
shape two equally exact algorithms agree in their root-mean-square error to a few
tenths of a percent."""

import math

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MARGIN = 1.01


def dct(n):
    k, m = torch.arange(n, device="cuda")[:, None], 2 * torch.arange(n, device="cuda")[None, :] + 1
    return torch.cos(((k * m) % (4 * n)).double() * (math.pi / (2 * n)))


def idct(n):
    d = dct(n).T * (2.0 / n)
    d[:, 0] *= 0.5
    return d


@pytest.mark.parametrize("shape", [(32, 32), (32, 512), (64, 32), (64, 64), (64, 256), (64, 512), (64, 2048), (128, 64),
                                   (256, 32), (512, 64), (1024, 64), (2048, 64)])
def test_error_of_default_against_two_sequence_kernels(shape):
    from paper_2110_01172_gb300 import Plan
    n1, n2 = shape
    batch = max(2, (1 << 20) // (n1 * n2))
    plans = [Plan(shape, batch=batch), Plan(shape, batch=batch, family="pair")]
    total = torch.zeros(2, 2, dtype=torch.float64)  # [direction][plan]
    for seed in range(3):
        gen = torch.Generator(device="cuda").manual_seed(seed)
        x = torch.rand((batch, n1, n2), generator=gen, device="cuda").mul_(2).sub_(1)
        spectrum = dct(n1) @ x.double() @ dct(n2).T
        c = spectrum.float()
        back = idct(n1) @ c.double() @ idct(n2).T
        for p, plan in enumerate(plans):
            total[0, p] += ((plan.forward(x).double() - spectrum).norm() / spectrum.norm()).item() ** 2
            total[1, p] += ((plan.inverse(c).double() - back).norm() / back.norm()).item() ** 2
    rms = (total / 3).sqrt()
    print(shape, rms.tolist())
    assert (rms[:, 0] <= MARGIN * rms[:, 1]).all()
