"""FOR, delta and RLE columns encoded by several threads per chunk (pieces of
65,536 rows): the library's bytes equal the oracle's at the row counts where a
piece ends, for runs across pieces, and for constant and extreme values."""
import numpy as np
import pytest

import oracle

zf = pytest.importorskip("paper_2602_08190_gb300")

P = 65536
SCHEMES = {"for": (zf.ZF_FOR_BP, oracle.FOR_BP), "delta": (zf.ZF_DELTA_BP, oracle.DELTA_BP), "rle": (zf.ZF_RLE, oracle.RLE)}


def _columns(n, dt):
    r = np.random.default_rng(n)
    lo, hi = np.iinfo(dt).min, np.iinfo(dt).max
    yield np.repeat(r.integers(-9, 9, n // 1000 + 1), 1000)[:n].astype(dt)      # runs across pieces
    yield np.full(n, 7, dt)                                                     # one run
    yield r.integers(lo, hi, n, dtype=dt)                                       # full width
    x = np.cumsum(r.integers(0, 5, n)).astype(dt)
    x[n // 2] = hi
    yield x


@pytest.mark.parametrize("scheme", SCHEMES)
@pytest.mark.parametrize("n", [1, P - 1, P, P + 1, 2 * P, 3 * P + 1025])
def test_bytes_equal_the_oracle(scheme, n):
    lib, orc = SCHEMES[scheme]
    for dt in (np.int32, np.int64):
        for x in _columns(n, dt):
            for chunk in (1 << 20, 3 * 32768):
                col = zf.Column(x)
                h = zf.zf_compress_host(zf.zf_plan(None, col, scheme=lib, chunk_rows=chunk), col)
                b = zf.zf_compressed_bytes(h)
                zf.zf_compressed_free(h)
                assert b == oracle.encode(x, orc, chunk)
