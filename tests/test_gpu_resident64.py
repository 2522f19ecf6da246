"""The FP64 resident time loop (automatic path, small grids) against the
single-step TMA kernel: the same arithmetic term for term, so bit for bit."""
import numpy as np
import pytest

from paper_1901_06503_gb300 import build_lib
from paper_1901_06503_gb300 import ffpat as F
from paper_1901_06503_gb300.inputs import random_speed, random_volume

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_lib.build()
    F.lib()
    yield
    F.set_stencil_path(0)


# 32 x 8 tiles with remainders in x and y, z-ranges of one plane (24 .. 40) to
# six (96), the last grid that fits and the first that does not (98); one, two,
# odd and even step counts
@pytest.mark.parametrize("n,T", [(4, 0.9), (6, 0.3), (24, 0.004), (24, 0.03), (32, 0.3),
                                 (34, 0.31), (40, 0.2), (64, 0.1), (90, 0.08), (96, 0.06),
                                 (98, 0.05)])
def test_bit_identical_to_single_steps(n, T):
    prob = F.problem(n, T, 4)
    c = torch.as_tensor(random_speed(n, n), device="cuda")
    h = torch.as_tensor(random_volume(n, n + 1), device="cuda")
    got = {}
    for path in (0, 2):
        F.set_stencil_path(path)
        got[path] = [F.wave(prob, c, h, transpose=t).cpu().numpy() for t in (False, True)]
        got[path].append(F.fb_solve(prob, c, F.project(prob, h), 1e-3, 0.2, 2)[0].cpu().numpy())
    F.set_stencil_path(0)
    assert F.device_status() == 0
    for a, b in zip(got[0], got[2]):
        assert np.isfinite(a).all() and np.array_equal(a, b)
