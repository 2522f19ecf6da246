"""The checkpoint buffer: 2 ceil(Nt / every) + every + 2 volumes are enough for every
problem; more is asked for only where there are segments to overlap."""
import numpy as np
import pytest

from paper_1901_06503_gb300 import build_lib
from paper_1901_06503_gb300 import ffpat as F
from paper_1901_06503_gb300.inputs import random_data, random_speed, random_volume


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_lib.build()


def least(prob, nt, every):
    n, es = prob.n, 8 if prob.precision == F.FP64 else 4
    row = n if es == 8 or n < 5 else (n + 3) // 4 * 4
    vol = (n * n * row * es + 255) // 256 * 256
    return (2 * (-(-nt // every)) + every + 2) * vol, vol


@pytest.mark.parametrize("prec", [F.FP64, F.FP32, F.FP32_KAHAN])
@pytest.mark.parametrize("n", [3, 8, 33, 64, 84, 85, 128])
def test_size(n, prec):
    prob = F.problem(n, 1.0, 8, prec)
    for nt, every in ((1, 1), (1, 4096), (10, 16), (16, 16), (17, 16), (31, 16), (100, 16),
                      (100, 1), (300, 299), (5000, 4096)):
        want, vol = least(prob, nt, every)
        overlap = prec != F.FP64 and n <= 84 and nt > every
        got = F.ckpt_bytes(prob, nt, every)
        assert got == want + (min(every, nt - every) * vol if overlap else 0), (nt, every)


@pytest.mark.gpu
@pytest.mark.parametrize("n,T,every", [(24, 0.3, 4), (33, 0.2, 8), (36, 0.4, 16), (64, 0.1, 20),
                                       (64, 0.1, 1000)])
def test_least_buffer(n, T, every):
    """The same bits as with the buffer that ffpat_ckpt_bytes asks for, nothing written
    behind it, and a byte less is refused."""
    torch = pytest.importorskip("torch")
    prob = F.problem(n, T, 6, F.FP32)
    c, h, w = (torch.as_tensor(a.astype(np.float32), device="cuda") for a in (
        random_speed(n, n), random_volume(n, n + 1), random_data(6, n, n + 2)))
    nt = F.problem_info(prob, float(c.max()))[0]
    size = least(prob, nt, every)[0]
    out = []
    for bytes_ in (F.ckpt_bytes(prob, nt, every), size):
        raw = torch.full((bytes_ + 4096,), 171, dtype=torch.uint8, device="cuda")
        ck = raw[:bytes_]
        g = F.forward_ckpt(prob, c, h, every, ck)
        out.append((g, *F.backward(prob, c, w, every, ck)))
        assert bool((raw[bytes_:] == 171).all())
    for a, b in zip(*out):
        assert torch.isfinite(a).all() and torch.equal(a, b)
    for call in (lambda ck: F.forward_ckpt(prob, c, h, every, ck),
                 lambda ck: F.backward(prob, c, w, every, ck)):
        with pytest.raises(F.FFPATError) as e:
            call(torch.empty(size - 1, dtype=torch.uint8, device="cuda"))
        assert e.value.code == F.ENOMEM
