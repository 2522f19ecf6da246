"""The checkpointed forward pass and the backward segments in the resident scheme
(FP32, automatic path, N <= 128) and on padded rows, against the step-by-step
loops: the same arithmetic in the same order, so bit for bit."""
import numpy as np
import pytest

from paper_1901_06503_gb300 import build_lib
from paper_1901_06503_gb300 import ffpat as F
from paper_1901_06503_gb300.autograd import forward_op
from paper_1901_06503_gb300.inputs import random_data, random_speed, random_volume

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_lib.build()
    F.lib()
    yield
    F.set_stencil_path(0)


def gradients(prob, c, h, w, every, path):
    F.set_stencil_path(path)
    try:
        ht, ct = (torch.tensor(a, device="cuda", dtype=torch.float32, requires_grad=True)
                  for a in (h, c))
        g = forward_op(ht, ct, prob, every)
        (g * w).sum().backward()
        torch.cuda.synchronize()
    finally:
        F.set_stencil_path(0)
    return [a.detach().cpu().numpy() for a in (g, ht.grad, ct.grad)]


# one step, one segment (every > Nt), segments of one and two steps, a last
# segment cut short; tiles with remainders; rows of every remainder mod 4 (n not a
# multiple of four: padded rows on every path, so against FP64 instead)
@pytest.mark.parametrize("n,T,every", [(24, 0.004, 4), (24, 0.03, 1), (24, 0.3, 2), (24, 0.3, 5),
                                       (36, 0.4, 16), (64, 0.2, 16), (68, 0.1, 7),
                                       (100, 0.06, 1000), (128, 0.05, 4)])
def test_segments_bit_identical(n, T, every):
    prob = F.problem(n, T, 6, F.FP32)
    c, h = random_speed(n, n).astype(np.float32), random_volume(n, n + 1).astype(np.float32)
    w = torch.tensor(random_data(6, n, n + 2), device="cuda", dtype=torch.float32)
    got, want = (gradients(prob, c, h, w, every, p) for p in (0, 2))
    assert F.device_status() == 0
    for a, b in zip(got, want):
        assert np.isfinite(a).all() and np.array_equal(a, b)


@pytest.mark.parametrize("prec", [F.FP32, F.FP32_KAHAN])
@pytest.mark.parametrize("n,T,every", [(5, 0.9, 3), (33, 0.1, 4), (66, 0.1, 16), (35, 0.15, 1),
                                       (131, 0.03, 4)])
def test_padded_rows(n, T, every, prec):
    """Against the FP64 operator at the FP32 inputs.  The gradient's last step is a
    difference of two fields that grow with the step count, 2e-5 for a few dozen."""
    prob, p64 = F.problem(n, T, 6, prec), F.problem(n, T, 6, F.FP64)
    c, h = random_speed(n, n).astype(np.float32), random_volume(n, n + 1).astype(np.float32)
    w = torch.tensor(random_data(6, n, n + 2), device="cuda", dtype=torch.float32)
    got = gradients(prob, c, h, w, every, 0)
    ht, ct = (torch.tensor(a, device="cuda", dtype=torch.float64, requires_grad=True)
              for a in (h, c))
    g = forward_op(ht, ct, p64, every)
    (g * w.double()).sum().backward()
    for a, b in zip(got, (g, ht.grad, ct.grad)):
        b = b.detach().cpu().numpy()
        assert np.linalg.norm(a - b) <= 2e-5 * np.linalg.norm(b)
    # a checkpoint buffer off the 16-byte grid takes the plain kernels: same bits
    nt, _, _ = F.problem_info(prob, float(c.max()))
    raw = torch.empty(F.ckpt_bytes(prob, nt, every) + 256, dtype=torch.uint8, device="cuda")
    cd, hd = torch.tensor(c, device="cuda"), torch.tensor(h, device="cuda")
    ck = raw[4:raw.numel() - 252]
    gg = F.forward_ckpt(prob, cd, hd, every, ck)
    gh, gc = F.backward(prob, cd, w, every, ck)
    for a, b in zip(got, (gg, gh, gc)):
        assert np.array_equal(a, b.cpu().numpy())
