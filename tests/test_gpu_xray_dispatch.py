"""P and P^T at every split of the work that their dispatch chooses, against the
oracle: rays of a CTA and warps a ray, voxel blocks of a CTA, planes a lane.
Tolerances as for the slab widths (tests/test_gpu_xray_slabs.py).
"""
import numpy as np
import pytest

import oracle.oracle as o
from paper_1901_06503_gb300 import build_lib
from paper_1901_06503_gb300 import ffpat as F
from paper_1901_06503_gb300.inputs import random_data, random_volume

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_lib.build()
    F.lib()


def rel(a, b):
    return float(np.linalg.norm((a - b).ravel()) / max(np.linalg.norm(b.ravel()), 1e-300))


# P: a ray by one warp of sixteen (from 4864 rays x slabs on), by two, by four; a last
# block of rays and of rows cut short in each
@pytest.mark.parametrize("n,nth", [(64, 90), (81, 61), (96, 52), (64, 45), (49, 70), (33, 2),
                                   (130, 7), (17, 9)])
def test_project_fp32(n, nth):
    p = random_volume(n, n).astype(np.float32)
    got = F.project(F.problem(n, 1.0, nth, F.FP32), torch.as_tensor(p, device="cuda"))
    assert rel(got.double().cpu().numpy(), o.project(p.astype(np.float64), nth)) < 5e-7


# P^T: CTAs of 4 x 2 blocks of 2 x 2 voxels (from 304 CTAs on), 2 x 2, 2 x 1 and 1 x 1;
# a last batch of eight angles cut short, one angle alone
@pytest.mark.parametrize("n,nth", [(128, 9), (131, 8), (96, 17), (97, 1), (64, 45), (67, 15),
                                   (32, 180), (21, 23), (3, 65)])
def test_backproject_fp32(n, nth):
    g = random_data(nth, n, n).astype(np.float32)
    got = F.backproject(F.problem(n, 1.0, nth, F.FP32), torch.as_tensor(g, device="cuda"))
    assert rel(got.double().cpu().numpy(), o.backproject(g.astype(np.float64), n)) < 5e-7


# FP64 P: one slab of one plane a lane (16, 12, 8 and 4 rays a CTA), one and two of two
# planes, three and four of one; P^T: one, two and four planes a lane, one block a CTA
# and four
@pytest.mark.parametrize("n,nth", [(30, 180), (28, 110), (28, 90), (25, 60), (24, 12), (64, 20), (100, 6),
                                   (90, 5), (129, 2), (66, 7), (128, 4), (160, 3), (73, 33)])
def test_fp64(n, nth):
    p, g = random_volume(n, n + 1), random_data(nth, n, n + 2)
    prob = F.problem(n, 1.0, nth, F.FP64)
    got = F.project(prob, torch.as_tensor(p, device="cuda")).cpu().numpy()
    assert np.array_equal(got, o.project(p, nth))
    got = F.backproject(prob, torch.as_tensor(g, device="cuda")).cpu().numpy()
    assert rel(got, o.backproject(g, n)) < 1e-12
