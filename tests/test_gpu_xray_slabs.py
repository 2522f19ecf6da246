"""P and P^T run along z in slabs of planes: the sizes where the slab width, the
lanes' vectors or the row blocks change or have a remainder, against the oracle.

Tolerances: the FP64 projection bit for bit and its transpose to 1e-12; FP32
5e-7 relative L2, that of the other FP32 projection tests (weights to about two
roundings, sums of at most 24 terms per eight rows and then N / 8 of those).
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


@pytest.mark.parametrize("n,nth", [(1, 2), (2, 3), (3, 5), (9, 4), (31, 7), (32, 5), (33, 2),
                                   (63, 3), (65, 8), (96, 3), (97, 2), (129, 5), (160, 3),
                                   (161, 2), (193, 3), (257, 2), (321, 3), (385, 2)])
def test_slab_widths_fp32(n, nth):
    prob = F.problem(n, 1.0, nth, F.FP32)
    p, g = (a.astype(np.float32) for a in (random_volume(n, 40 + n), random_data(nth, n, 50 + n)))
    got = F.project(prob, torch.as_tensor(p, device="cuda")).double().cpu().numpy()
    assert rel(got, o.project(p.astype(np.float64), nth)) < 5e-7
    got = F.backproject(prob, torch.as_tensor(g, device="cuda")).double().cpu().numpy()
    assert rel(got, o.backproject(g.astype(np.float64), n)) < 5e-7


@pytest.mark.parametrize("n,nth", [(1, 2), (2, 3), (3, 5), (9, 40), (31, 7), (33, 2), (64, 3),
                                   (65, 33), (97, 2), (129, 5), (257, 2)])
def test_slab_widths_fp64(n, nth):
    prob = F.problem(n, 1.0, nth, F.FP64)
    p, g = random_volume(n, 60 + n), random_data(nth, n, 70 + n)
    got = F.project(prob, torch.as_tensor(p, device="cuda")).cpu().numpy()
    assert np.array_equal(got, o.project(p, nth))
    got = F.backproject(prob, torch.as_tensor(g, device="cuda")).cpu().numpy()
    assert rel(got, o.backproject(g, n)) < 1e-12


# Lambda: 32 rows a CTA, 16 outputs of one parity a warp, 512 inputs at a time,
# outputs over several CTAs beyond 256
@pytest.mark.parametrize("n,nth", [(1, 3), (2, 1), (3, 5), (63, 1), (65, 2), (66, 3), (127, 1),
                                   (193, 1), (257, 1), (385, 1), (511, 1), (514, 1), (1030, 1)])
def test_ramp_shapes(n, nth):
    rows = random_data(nth, n, 80 + n)
    for prec, dt, tol in ((F.FP64, np.float64, 1e-12), (F.FP32, np.float32, 5e-7)):
        prob = F.problem(n, 1.0, nth, prec)
        r = rows.astype(dt)
        got = F.ramp(prob, torch.as_tensor(r, device="cuda")).double().cpu().numpy()
        assert rel(got, o.ramp(r.astype(np.float64))) < tol


# standalone calls take operands beyond 1 GiB in several passes over z: P in two at
# 656^3 FP32 (384 planes and 272) and 520^3 FP64 (480 and 40), P^T in two or more with
# that many rows of data.  The planes are independent: with the planes moved by half
# the grid every result moves with them, out of one pass into another; rays of every
# pass are checked against the oracle too.
@pytest.mark.parametrize("n,prec", [(656, F.FP32), (520, F.FP64)])
def test_passes_over_z(n, prec):
    dt = torch.float64 if prec == F.FP64 else torch.float32
    gen = torch.Generator(device="cuda").manual_seed(n)
    tol = 1e-12 if prec == F.FP64 else 5e-7

    def off(a, b):
        return float((a.double() - b.double()).norm() / b.double().norm())

    prob = F.problem(n, 1.0, 2, prec)
    p = torch.randn((n, n, n), generator=gen, device="cuda", dtype=dt)
    got = F.project(prob, p)
    assert off(F.project(prob, p.roll(n // 2, 0)).roll(-(n // 2), 1), got) < tol
    jlk = [(j, z, k) for j in (0, 1) for z in (0, 383, 384, 479, 480, n - 1)
           for k in range(0, n, 37)]
    want = o.project_rays(p.double().cpu().numpy(), 2, jlk)
    have = np.array([got[t].item() for t in jlk])
    assert rel(have, want) < tol
    del p, got
    nth = 2 * n if prec == F.FP32 else 520
    prob = F.problem(n, 1.0, nth, prec)
    g = torch.randn((nth, n, n), generator=gen, device="cuda", dtype=dt)
    got = F.backproject(prob, g)
    assert off(F.backproject(prob, g.roll(n // 2, 1)).roll(-(n // 2), 0), got) < tol


# P of a smooth volume, where the rows' sums all have one sign: the error of a long
# plain sum would grow with N.  Expected at most 8e-8: the rounded cell size (6e-8
# where 2 / N is no power of two), the last addition and the product (3.4e-8 each)
# and the groups of eight rows (24 additions each, N / 8 of them averaged: 2e-8).
@pytest.mark.parametrize("n,nth", [(32, 4), (64, 3), (100, 4), (150, 4), (256, 2)])
def test_smooth_sums(n, nth):
    x = np.linspace(-1, 1, n)
    p = np.exp(-4 * ((x - 0.1) ** 2 + (x[:, None] + 0.2) ** 2 + x[:, None, None] ** 2))
    p = p.astype(np.float32)
    got = F.project(F.problem(n, 1.0, nth, F.FP32), torch.as_tensor(p, device="cuda"))
    assert rel(got.double().cpu().numpy(), o.project(p.astype(np.float64), nth)) < 8e-8


# sums beyond the largest float are infinite, not NaN
def test_overflow_stays_infinite():
    p = torch.full((64, 64, 64), 3e38, device="cuda")
    g = F.project(F.problem(64, 1.0, 4, F.FP32), p)
    assert not torch.isnan(g).any() and torch.isinf(g[:, :, 32]).all()
