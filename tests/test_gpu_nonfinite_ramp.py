"""An infinite detector value stays infinite through Lambda: the outputs its odd
taps (and t_0) reach are +-inf, the others are those of the row without it, bit
for bit (no tap reaches them)."""
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


# inputs in one stage and in several (beyond 512), outputs over several CTAs (beyond 256)
@pytest.mark.parametrize("prec", [F.FP64, F.FP32])
@pytest.mark.parametrize("n", [2, 33, 64, 300, 600])
def test_infinite_detector(n, prec):
    prob = F.problem(n, 1.0, 2, prec)
    r = torch.as_tensor(random_data(2, n, n), device="cuda").to(F.torch_dtype(prob))
    at = [(0, 0, 0), (0, n - 1, n - 1), (1, 0, n // 2), (1, 1, min(3, n - 1))]
    k = np.arange(n)
    for sign in (1.0, -1.0):
        zeroed, spoilt = r.clone(), r.clone()
        for i in at:
            zeroed[i], spoilt[i] = 0.0, sign * np.inf
        want = F.ramp(prob, zeroed).cpu().numpy()
        for j, z, x in at:
            want[j, z, (k - x) % 2 == 1] = -sign * np.inf
            want[j, z, x] = sign * np.inf
        assert np.array_equal(F.ramp(prob, spoilt).cpu().numpy(), want)
