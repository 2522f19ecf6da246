"""P^T of data with an infinite value: infinite in the voxels that see it, and in
all others, bit for bit, what the data without it give."""
import numpy as np
import pytest

from paper_1901_06503_gb300 import build_lib
from paper_1901_06503_gb300 import ffpat as F
from paper_1901_06503_gb300.inputs import random_data

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_lib.build()
    F.lib()


@pytest.mark.parametrize("prec", [F.FP64, F.FP32])
@pytest.mark.parametrize("n,nth", [(7, 3), (33, 10), (64, 9), (150, 4), (300, 3)])
def test_infinite_datum(n, nth, prec):
    prob = F.problem(n, 1.0, nth, prec)
    g = torch.as_tensor(random_data(nth, n, n), device="cuda").to(F.torch_dtype(prob))
    at = [(0, 0, n // 2), (1, n // 2, n // 3), (nth - 1, n - 1, n - 1)]
    seen = torch.zeros_like(g)
    zeroed, spoilt = g.clone(), g.clone()
    for i in at:
        seen[i], zeroed[i], spoilt[i] = 1.0, 0.0, np.inf
    seen = F.backproject(prob, seen) != 0
    assert seen.any() and not seen.all()
    want = F.backproject(prob, zeroed)
    want[seen] = np.inf
    assert torch.equal(F.backproject(prob, spoilt), want)
