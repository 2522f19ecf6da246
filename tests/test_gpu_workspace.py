"""The workspace's volumes serve several operands one after the other (P and P^T's
z-innermost copies and, on ragged grids, Lambda's result lie in the state volumes).

Every call against the same steps as calls of their own, each with its own
workspace: FP64 1e-12 relative L2 (the scalings round in another order), FP32
2e-6 (a few roundings of either side, amplified by at most the norm of one
operator).  And every call on a workspace that holds NaN against one that holds
zeros, bit for bit: nothing is read before it is written.
"""
import math

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


def dev(prob, a):
    return torch.as_tensor(a, device="cuda").to(F.torch_dtype(prob))


def off(a, b):
    return float((a.double() - b.double()).norm() / b.double().norm())


# ragged and aligned rows; data that fit beside Lambda's result in the state volumes,
# data that do not, and more than the state and one data array hold with z innermost
@pytest.mark.parametrize("prec", [F.FP64, F.FP32, F.FP32_KAHAN])
@pytest.mark.parametrize("n,pad,nth", [(34, 0, 6), (34, 0, 100), (33, 0, 400), (64, 0, 24),
                                       (36, 0, 300), (25, 5, 9), (24, 4, 70), (12, 0, 90),
                                       (129, 0, 3)])
def test_shared_volumes(n, pad, nth, prec):
    nw, T = n + 2 * pad, 6.0 / n
    tol = 1e-12 if prec == F.FP64 else 2e-6
    for precond in (F.PRECOND_NONE, F.PRECOND_RAMP):
        prob = F.problem(n, T, nth, prec, precond, pad=pad)
        c, h = dev(prob, random_speed(nw, n)), dev(prob, np.abs(random_volume(n, n + 1)))
        g = dev(prob, random_data(nth, nw, n + 2))
        step, lam = 0.1, 1e-3

        assert off(F.forward(prob, c, h), F.project(prob, F.wave(prob, c, h))) < tol

        def adjoint(q):
            return F.wave(prob, c, F.backproject(prob, q), transpose=True)
        assert off(F.adjoint(prob, c, g), adjoint(g)) < tol
        scale = 2 * math.pi / (nth * 2 / n)
        assert off(F.fbp(prob, g), F.backproject(prob, F.ramp(prob, g)) * scale) < tol
        r = F.project(prob, F.wave(prob, c, h)) - g
        lr = F.ramp(prob, r) if precond == F.PRECOND_RAMP else r
        want = (h - step * adjoint(lr) - step * lam).clamp_min(0.0)
        got, _, hist = F.fb_solve(prob, c, g, lam, step, 1, h=h.clone())
        assert off(got, want) < tol
        objective = 0.5 * float((lr.double() * r.double()).sum()) + lam * float(h.double().sum())
        assert abs(hist[0, 0] - objective) < 1e3 * tol * abs(objective)
        assert abs(hist[0, 1] - float(r.double().norm())) < tol * hist[0, 1]


@pytest.mark.parametrize("prec", [F.FP64, F.FP32, F.FP32_KAHAN])
@pytest.mark.parametrize("n,pad,nth", [(33, 0, 7), (34, 0, 50), (64, 0, 9), (21, 5, 4),
                                       (130, 0, 2)])
def test_contents_on_entry_do_not_matter(n, pad, nth, prec):
    nw = n + 2 * pad
    prob = F.problem(n, 6.0 / n, nth, prec, F.PRECOND_RAMP, pad=pad)
    c, h, q = (dev(prob, a) for a in (random_speed(nw, n), random_volume(n, 1),
                                      random_volume(nw, 2)))
    g = dev(prob, random_data(nth, nw, 3))
    calls = [
        lambda ws: F.forward(prob, c, h, ws=ws), lambda ws: F.adjoint(prob, c, g, ws=ws),
        lambda ws: F.wave(prob, c, h, ws=ws), lambda ws: F.wave(prob, c, q, transpose=True, ws=ws),
        lambda ws: F.fbp(prob, g, ws=ws),
        lambda ws: torch.tensor(F.opnorm(prob, c, h, 2, ws=ws)),
        lambda ws: F.fb_solve(prob, c, g, 1e-3, 0.1, 2, ws=ws)[0],
        lambda ws: F.fb_solve_masked(prob, c, g, 1e-3, 0.1, 2, ws=ws, reg=F.REG_GRAD2)[0],
        lambda ws: F.fb_two_step(prob, c, g, 1e-3, 0.1, 2, ws=ws)[0],
        lambda ws: F.fb_two_step(prob, c, g, 1e-3, 0.1, 2, ws=ws, reg=F.REG_GRAD2)[0]]
    if pad == 0:
        nt = F.problem_info(prob, float(c.max()))[0]

        def gradients(ws):
            ckpt = torch.empty(F.ckpt_bytes(prob, nt, 4), dtype=torch.uint8, device="cuda")
            ckpt.fill_(int(ws[0]))
            out = F.forward_ckpt(prob, c, h, 4, ckpt, ws=ws)
            ws.fill_(int(ws[-1]))
            return torch.cat([t.flatten() for t in (out, *F.backward(prob, c, g, 4, ckpt, ws=ws))])
        calls.append(gradients)
    for i, call in enumerate(calls):
        out = []
        for byte in (0, 255):  # doubles and floats of 0xff bytes are NaN
            ws = F.workspace(prob)
            ws.fill_(byte)
            out.append(call(ws))
        assert torch.isfinite(out[0]).all() and torch.equal(out[0], out[1]), i
