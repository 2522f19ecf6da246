"""ffpat_workspace_bytes: no more than the dense volumes and data that the methods
work on, whatever layouts the kernels keep beside them (host only)."""
import pytest

from paper_1901_06503_gb300 import build_lib
from paper_1901_06503_gb300 import ffpat as F


def up(b):
    return (b + 255) // 256 * 256


def dense(n, pad, nth, prec):
    """kappa, two image volumes, the wavefield state, two data arrays, the padded
    grid's kappa, input, FBP volume and box result, and the small tables."""
    es = 8 if prec == F.FP64 else 4
    nw, k = n + 2 * pad, {F.FP64: 2, F.FP32: 4, F.FP32_KAHAN: 6}[prec]
    vol, wav, dat = up(n**3 * es), up(nw**3 * es), up(nth * nw**2 * es)
    b = 3 * vol + k * wav + 2 * dat + (3 * wav + vol if pad else 0)
    return b + up(8 * 8 * 608) + up(8 * 64) + up(8 * 8 * 4096) + up(32 * nth) + up(
        2 * n * n * es + 8 * n) + 128 * 1024


def padding(nw, prec):
    """Elements that rows of a multiple of 16 bytes add to a row."""
    return -nw % (2 if prec == F.FP64 else 4)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_lib.build()


SIZES = [*range(32, 72), 95, 96, 97, 100, 101, 127, 128, 129, 130, 150, 161, 192, 196, 200, 257,
         300, 321, 384, 388, 400, 513, 1000, 1499, 2048]


@pytest.mark.parametrize("prec", [F.FP64, F.FP32, F.FP32_KAHAN])
@pytest.mark.parametrize("pad", [0, 1, 5, 64])
def test_no_more_than_dense(prec, pad):
    for n in SIZES:
        nw = n + 2 * pad
        for nth in (25, 33, 45, 90, 180, 1000, 65535):
            ragged = padding(nw, prec)
            got, most = F.workspace_bytes(F.problem(n, 1.0, nth, prec, pad=pad)), dense(
                n, pad, nth, prec)
            if not ragged or nth <= nw:
                assert got <= most, (n, nth)
            else:  # more angles than the state volumes hold: the padding of the rows
                assert got <= most + 9 * (ragged * nw * nw * 8 + 256), (n, nth)


@pytest.mark.parametrize("prec", [F.FP64, F.FP32, F.FP32_KAHAN])
def test_small_grids_and_few_angles(prec):
    """Below 32 points a slab of 32 planes each for the wave input and the data;
    with few angles on ragged rows the padding of at most nine volumes."""
    es = 8 if prec == F.FP64 else 4
    for n in range(1, 32):
        for nth in (1, 7, 180, 65535):
            got = F.workspace_bytes(F.problem(n, 1.0, nth, prec))
            slabs = 32 * n * (n + 2 * nth) * es + 9 * (padding(n, prec) * n * n * es + 512)
            assert got <= dense(n, 0, nth, prec) + slabs, (n, nth)
    for n in SIZES:
        for nth in (1, 7, 24):
            got = F.workspace_bytes(F.problem(n, 1.0, nth, prec))
            assert got <= dense(n, 0, nth, prec) + 9 * padding(n, prec) * n * n * es, (n, nth)
