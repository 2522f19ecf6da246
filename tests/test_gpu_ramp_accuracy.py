"""Lambda of smooth rows in FP32 is as close to 64 bits as the sum from t_0 outwards,
pair by pair, in FP32: there the terms cancel from the largest on, so every later
addition rounds at the size of what is left.  (Plain rounding analysis; 2 % for the
last bits that a fused multiply-add may round otherwise.)
"""
import numpy as np
import pytest

from paper_1901_06503_gb300 import build_lib
from paper_1901_06503_gb300 import ffpat as F

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def rows(n, count):
    """Spherical-wave profiles of a few blobs."""
    rng = np.random.default_rng(n)
    x = (np.arange(n) + 0.5) * 2 / n - 1
    r = np.zeros((count, n))
    for q in range(count):
        for _ in range(4):
            u = np.abs(x - rng.uniform(-0.6, 0.6))
            a, b, s = rng.uniform(0.3, 1), rng.uniform(0.1, 0.9), 0.08

            def wave(v):
                return v * np.exp(-v**2 / (2 * s * s))
            r[q] += a * (wave(u - b) + wave(u + b))
    return r.astype(np.float32)


def taps(n):
    d = np.arange(n, dtype=float)
    t = np.zeros(n)
    t[0], t[1::2] = n / 16, -n / (4 * np.pi**2 * d[1::2] ** 2)
    return t


def outwards(r):
    n = r.shape[1]
    t = taps(n).astype(np.float32)
    p = np.pad(r, ((0, 0), (n, n)))
    acc = t[0] * r
    for d in range(1, n, 2):
        pair = (p[:, n - d:2 * n - d] + p[:, n + d:2 * n + d]).astype(np.float64)
        acc = (t[d].astype(np.float64) * pair + acc).astype(np.float32)  # fused
    return acc


@pytest.mark.parametrize("n", [64, 192, 256, 300, 384, 448, 512, 768, 1024])
def test_smooth_rows(n):
    build_lib.build()
    r = rows(n, n)
    k = np.arange(n)
    want = r.astype(np.float64) @ taps(n)[np.abs(k[:, None] - k[None, :])]
    prob = F.problem(n, 1.0, 1, F.FP32)
    got = F.ramp(prob, torch.as_tensor(r[None], device="cuda"))[0].cpu().numpy()
    off = [np.linalg.norm(a - want) / np.linalg.norm(want) for a in (got, outwards(r))]
    assert off[0] <= 1.02 * off[1], off
