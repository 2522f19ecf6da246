"""ffpat_project and ffpat_backproject where little device memory is to be had: they
work in narrower passes over z instead of failing.

The library allocates from the device's current memory pool; a pool of at most 48
MiB (wave grids whose z-innermost operand takes 130 MB and more) stands for a full
device.  The slabs differ, so the order of P's sums may: 5e-7 relative L2 in FP32 and
1e-12 in FP64, as for passes over z elsewhere.
"""
import contextlib
import ctypes

import pytest

from paper_1901_06503_gb300 import build_lib
from paper_1901_06503_gb300 import ffpat as F

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


class PoolProps(ctypes.Structure):  # CUmemPoolProps
    _fields_ = [("alloc_type", ctypes.c_int), ("handle_types", ctypes.c_int),
                ("location_type", ctypes.c_int), ("location_id", ctypes.c_int),
                ("security", ctypes.c_void_p), ("max_size", ctypes.c_size_t),
                ("usage", ctypes.c_ushort), ("reserved", ctypes.c_ubyte * 54)]


@contextlib.contextmanager
def pool_of(size):
    """The device's memory pool is one of at most `size` bytes."""
    cu = ctypes.CDLL("libcuda.so.1")

    def ok(rc):
        assert rc == 0, rc
    torch.cuda.synchronize()
    pool, default = ctypes.c_void_p(), ctypes.c_void_p()
    dev = torch.cuda.current_device()
    ok(cu.cuDeviceGetDefaultMemPool(ctypes.byref(default), dev))
    props = PoolProps(1, 0, 1, dev, None, size, 0)  # pinned, on the device
    ok(cu.cuMemPoolCreate(ctypes.byref(pool), ctypes.byref(props)))
    try:
        ok(cu.cuDeviceSetMemPool(dev, pool))
        yield
    finally:
        torch.cuda.synchronize()
        ok(cu.cuDeviceSetMemPool(dev, default))
        ok(cu.cuMemPoolDestroy(pool))


@pytest.mark.parametrize("n,nth,prec", [(321, 320, F.FP32), (400, 260, F.FP32), (257, 256, F.FP64)])
def test_narrower_passes(n, nth, prec):
    build_lib.build()
    gen = torch.Generator(device="cuda").manual_seed(n)
    prob = F.problem(n, 1.0, nth, prec)
    dt, tol = F.torch_dtype(prob), 1e-12 if prec == F.FP64 else 5e-7
    p = torch.randn((n, n, n), generator=gen, device="cuda", dtype=dt)
    g = torch.randn((nth, n, n), generator=gen, device="cuda", dtype=dt)
    want = F.project(prob, p), F.backproject(prob, g)
    have = torch.full_like(want[0], float("nan")), torch.full_like(want[1], float("nan"))
    with pool_of(48 << 20):
        F.project(prob, p, g=have[0])
        F.backproject(prob, g, h=have[1])
    for a, b in zip(have, want):
        assert float((a - b).double().norm() / b.double().norm()) < tol


def test_not_even_one_pass():
    """An error that does not stick: 32 planes of 1000^3 (128 MB) have no room."""
    prob = F.problem(1000, 1.0, 1, F.FP32)
    p = torch.ones((1000, 1000, 1000), device="cuda")
    with pool_of(48 << 20), pytest.raises(F.FFPATError) as e:
        F.project(prob, p)
    assert e.value.code == F.ECUDA and "out of memory" in str(e.value)
    assert torch.isfinite(F.project(prob, p)).all()
