"""Grids whose rows are no multiple of 16 bytes run on padded rows (automatic
path): the same results as the plain kernel on the rows as they are.

FP32 and FP32-Kahan steps agree bit for bit between the kernels; in FP64 they
differ in the rounding order of the Laplacian (1e-12 relative L2 for at most a
few hundred steps of a bounded recurrence).
"""
import numpy as np
import pytest

from paper_1901_06503_gb300 import build_lib
from paper_1901_06503_gb300 import ffpat as F
from paper_1901_06503_gb300.inputs import random_data, random_speed, random_volume

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_lib.build()
    F.lib()
    yield
    F.set_stencil_path(0)


def both(f):
    """f() on the automatic path and with the plain kernel."""
    out = []
    for path in (0, 1):
        F.set_stencil_path(path)
        r = f()
        torch.cuda.synchronize()
        out.append(r.double().cpu().numpy())
    F.set_stencil_path(0)
    return out


def check(f, prec):
    a, b = both(f)
    assert np.isfinite(a).all()
    if prec == F.FP64:
        assert np.linalg.norm(a - b) <= 1e-12 * np.linalg.norm(b)
    else:
        assert np.array_equal(a, b)


# one short of, on and past the 64-wide tiles, every remainder of n mod 4, the
# resident loop's range (to 128) and the two-step passes beyond it
@pytest.mark.parametrize("prec", [F.FP64, F.FP32, F.FP32_KAHAN])
@pytest.mark.parametrize("n,pad,T", [(5, 0, 0.9), (6, 0, 0.6), (7, 1, 0.6), (33, 0, 0.2),
                                     (63, 0, 0.1), (65, 0, 0.1), (66, 0, 0.1), (101, 0, 0.07),
                                     (127, 0, 0.05), (131, 0, 0.05), (134, 0, 0.045),
                                     (21, 5, 0.4)])
def test_padded_rows(n, pad, T, prec):
    prob = F.problem(n, T, 6, prec, pad=pad)
    nw = n + 2 * pad
    dev = lambda a: torch.as_tensor(a, device="cuda").to(F.torch_dtype(prob))  # noqa: E731
    c = dev(random_speed(nw, n))
    h, q, g = dev(random_volume(n, n + 1)), dev(random_volume(nw, n + 2)), dev(
        random_data(6, nw, n + 3))
    check(lambda: F.wave(prob, c, h), prec)
    check(lambda: F.wave(prob, c, q, transpose=True), prec)
    check(lambda: F.forward(prob, c, h), prec)
    check(lambda: F.adjoint(prob, c, g), prec)
    if pad == 0:
        # in place, from an unaligned address
        buf = torch.empty(n**3 + 1, dtype=h.dtype, device="cuda")
        box = buf[1:].view(n, n, n)

        def in_place():
            box.copy_(h)
            return F.wave(prob, c, box, out=box).clone()
        check(in_place, prec)


@pytest.mark.parametrize("prec", [F.FP64, F.FP32_KAHAN])
@pytest.mark.parametrize("n,pad,reg", [(34, 0, 0), (35, 0, 1), (25, 4, 1)])
def test_padded_rows_solves(n, pad, reg, prec):
    prob = F.problem(n, 0.3, 5, prec, F.PRECOND_RAMP, pad=pad)
    nw = n + 2 * pad
    dev = lambda a: torch.as_tensor(a, device="cuda").to(F.torch_dtype(prob))  # noqa: E731
    c, g = dev(random_speed(nw, n)), dev(random_data(5, nw, n + 3))
    check(lambda: F.fb_solve_masked(prob, c, g, 1e-3, 0.3, 3, reg=reg)[0], prec)
    check(lambda: F.fb_two_step(prob, c, g, 1e-3, 0.3, 3, reg=reg)[0], prec)
    v = dev(random_volume(n, 9))
    check(lambda: torch.tensor([F.opnorm(prob, c, v, 3)], dtype=torch.float64), F.FP64)
