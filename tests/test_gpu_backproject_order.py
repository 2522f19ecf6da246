"""P^T adds the angles in an order whose partial sums stay small where the data
change sign slowly with the angle (as filtered data do).

Data of one sign for the first half of the angles and of the other for the second:
with the angles in their own order the sum grows to n_angles / 2 contributions
before it falls, and each of the about 2.3 n_angles multiply-adds rounds at that
size.  Spread over the directions it stays within a batch's four contributions.
Expected in units of one angle's contribution w = dx (r.m.s.): additions
sqrt(2.3 * 180) * 0.29 * 2^-23 * 4 = 2.8e-6 at most, weights of two roundings each
sqrt(180) * 1e-7 = 1.3e-6, so 3.1e-6 at most; in angle order
sqrt(2.3 * 180) * 0.29 * 2^-23 * 50 = 3.5e-5.
"""
import pytest

from paper_1901_06503_gb300 import build_lib
from paper_1901_06503_gb300 import ffpat as F

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [33, 64, 130])
def test_angles_spread_over_the_directions(n):
    build_lib.build()
    nth = 180
    gen = torch.Generator(device="cuda").manual_seed(n)
    g = 0.5 + 0.5 * torch.rand((1, n, 1), generator=gen, device="cuda")
    g = g.expand(nth, n, n).clone()
    g[nth // 2:] *= -1.0
    got = F.backproject(F.problem(n, 1.0, nth, F.FP32), g).double()
    want = F.backproject(F.problem(n, 1.0, nth, F.FP64), g.double())
    err = (got - want)[:, n // 4:n - n // 4, n // 4:n - n // 4]
    assert float(err.square().mean().sqrt()) * n / 2 < 4e-6
