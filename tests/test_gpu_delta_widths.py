"""Delta blocks at every difference width and at the row counts where a step
of 128 values, a block of 1,024 or a chunk ends, ascending and descending and
with differences around the 32-bit offset path's limit, against the column."""
import numpy as np
import pytest

from gpu_helpers import Gpu, compress, out_specs

zf = pytest.importorskip("paper_2602_08190_gb300")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    g = Gpu()
    yield g
    g.close()


def _check(gpu, x, chunk=4096):
    h = compress(x, zf.ZF_DELTA_BP, chunk)
    try:
        for resident in (False, True):
            got, = gpu.decode([h], out_specs(x), resident=resident)
            assert np.array_equal(got, x)
    finally:
        zf.zf_compressed_free(h)


@pytest.mark.parametrize("bits", list(range(0, 34)) + [40, 47, 48, 63, 64])
def test_widths(gpu, bits):
    r = np.random.default_rng(bits)
    d = r.integers(0, 1 << bits, 5000, dtype=np.uint64) if bits < 64 else r.integers(0, 1 << 63, 5000, dtype=np.uint64) * np.uint64(2)
    d[1::1024] = 0                                      # every block reaches both ends of the width
    d[2::1024] = (1 << bits) - 1
    with np.errstate(over="ignore"):
        _check(gpu, np.cumsum(d, dtype=np.uint64).view(np.int64))
        if bits <= 32:
            _check(gpu, np.cumsum(d, dtype=np.uint64).astype(np.uint32).view(np.int32))


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 127, 128, 129, 131, 1023, 1024, 1025, 1027, 4095, 4097, 8191])
def test_row_counts(gpu, n):
    r = np.random.default_rng(n)
    for dt in (np.int32, np.int64):
        _check(gpu, np.cumsum(r.integers(-50, 50, n)).astype(dt))


@pytest.mark.parametrize("step", [(1 << 21) - 1, 1 << 21, (1 << 32) - 1, 1 << 40, -1, -(1 << 21), -(1 << 40)])
def test_smallest_differences(gpu, step):
    r = np.random.default_rng(5)
    _check(gpu, np.cumsum(step + r.integers(0, 1 << 21, 3000)))
    if abs(step) < 1 << 31:
        with np.errstate(over="ignore"):
            _check(gpu, np.cumsum(step + r.integers(0, 9, 3000)).astype(np.int32))
