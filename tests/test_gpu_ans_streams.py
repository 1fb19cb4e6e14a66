"""ANS decode at the sizes where a lane's window and ring of stream bytes can go
wrong: streams of every alignment, of four bytes only, with zero, one and two
bytes per row, alphabets on both sides of the slot entry's two layouts (128
symbols), and row counts that leave every remainder of a 32-byte store."""
import numpy as np
import pytest

from gpu_helpers import Gpu, out_specs

zf = pytest.importorskip("paper_2602_08190_gb300")
pytestmark = pytest.mark.gpu


def _skewed(r, n, nd, share):
    """`share` of the rows hold one value, the others are uniform over nd values."""
    x = r.integers(0, nd, n)
    x[r.random(n) < share] = 0
    x[: min(n, nd)] = np.arange(nd)[:n]
    return x


@pytest.mark.parametrize("nd", [1, 2, 4, 5, 127, 128, 129, 256])
@pytest.mark.parametrize("dt", [np.int32, np.int64])
def test_alphabets(nd, dt):
    r = np.random.default_rng(nd)
    vals = r.integers(-(1 << 31), (1 << 31) - 1, nd) if dt == np.int32 else r.integers(-(1 << 62), 1 << 62, nd)
    g = Gpu()
    try:
        for n, share, stream in ((40_003, 0.0, 512), (9_001, 0.99, 128), (5_005, 0.5, 32), (20_002, 0.9, 4096), (7, 0.0, 512)):
            x = vals[_skewed(r, n, nd, share)].astype(dt)
            col = zf.Column(x)
            h = zf.zf_compress_host(zf.zf_plan(None, col, scheme=zf.ZF_ANS, chunk_rows=16384, ans_stream_rows=stream), col)
            for resident in (False, True):
                got, = g.decode([h], out_specs(x), resident=resident)
                assert np.array_equal(got, x)
            zf.zf_compressed_free(h)
    finally:
        g.close()


def test_every_remainder_of_a_store():
    g = Gpu()
    try:
        for n in range(1, 27):
            x = (np.arange(n) % 3).astype(np.int32)
            col = zf.Column(x)
            h = zf.zf_compress_host(zf.zf_plan(None, col, scheme=zf.ZF_ANS, chunk_rows=1024, ans_stream_rows=32), col)
            got, = g.decode([h], out_specs(x))
            assert np.array_equal(got, x)
            zf.zf_compressed_free(h)
    finally:
        g.close()
