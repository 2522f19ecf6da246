"""Cooperative launches (the FP64 resident loop, the segments of the differentiated
operator) on two streams and from two host threads at once: results of one stream,
and no bounded wait runs out."""
import threading

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


def forward64(n, seed):
    prob = F.problem(n, 0.5, 8, F.FP64)
    c, h = (torch.as_tensor(a, device="cuda") for a in (random_speed(n, seed),
                                                        random_volume(n, seed + 1)))
    ws = F.workspace(prob)
    return lambda: (F.forward(prob, c, h, ws=ws),)


def gradients(n, seed):
    prob = F.problem(n, 0.3, 8, F.FP32)
    c, h, w = (torch.as_tensor(a, device="cuda").float() for a in (
        random_speed(n, seed), random_volume(n, seed + 1), random_data(8, n, seed + 2)))
    nt = F.problem_info(prob, float(c.max()))[0]
    ck = torch.empty(F.ckpt_bytes(prob, nt, 8), dtype=torch.uint8, device="cuda")
    ws = F.workspace(prob)
    return lambda: (F.forward_ckpt(prob, c, h, 8, ck, ws=ws), *F.backward(prob, c, w, 8, ck, ws=ws))


@pytest.mark.parametrize("make,sizes", [(forward64, (32, 96)), (gradients, (32, 84)),
                                        (gradients, (64, 64))])
def test_two_streams(make, sizes):
    calls = [make(n, 10 + i) for i, n in enumerate(sizes)]
    want = [call() for call in calls]
    torch.cuda.synchronize()
    got, errors = [None, None], []

    def work(i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(4):
                    got[i] = calls[i]()
                torch.cuda.current_stream().synchronize()
        except Exception as e:  # noqa: BLE001 (reported by the test)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors and F.device_status() == 0
    for a, b in zip(got, want):
        for x, y in zip(a, b):
            assert torch.isfinite(x).all() and torch.equal(x, y)
