"""zf_decompress_device_noalloc over the forms its one launch accepts: odd row
counts around tiles, jobs and chunks, widths whose staging buffers fit a CTA
four times, twice or once, every scheme and type, and malformed columns."""
import struct

import numpy as np
import pytest

import zf_workloads as W
from gpu_helpers import SENTINEL, compress

zf = pytest.importorskip("paper_2602_08190_gb300")
pytestmark = pytest.mark.gpu


def _wide(n, bits, dt):
    """n values spanning exactly `bits` bits (0: a constant)."""
    r = np.random.default_rng(n + bits)
    x = r.integers(0, 1 << bits, n, dtype=np.uint64) if bits < 64 else r.integers(0, 1 << 63, n, dtype=np.uint64) * np.uint64(2)
    if n > 1 and bits:
        x[0], x[-1] = 0, (1 << bits) - 1
    return x.view(np.int64).astype(dt)


COLUMNS = {
    "one row": (lambda: np.array([7], np.int32), zf.ZF_FOR_BP, 1024),
    "constant": (lambda: _wide(5000, 0, np.int64), zf.ZF_FOR_BP, 2048),
    "one row past a tile": (lambda: _wide(1025, 12, np.int32), zf.ZF_FOR_BP, 1024),
    "short last chunk": (lambda: _wide(3 * 5120 + 1, 31, np.int32), zf.ZF_FOR_BP, 5120),
    "full width, 32 bits": (lambda: _wide(70_001, 32, np.int32), zf.ZF_FOR_BP, 65536),
    "28 bits, four warps at once": (lambda: _wide(20_000, 28, np.int64), zf.ZF_FOR_BP, 8192),
    "48 bits, two warps at once": (lambda: _wide(20_000, 48, np.int64), zf.ZF_FOR_BP, 8192),
    "full width, 64 bits": (lambda: _wide(20_000, 64, np.int64), zf.ZF_FOR_BP, 8192),
    "dictionary of one": (lambda: np.full(3000, -5, np.int64), zf.ZF_DICT_BP, 1024),
    "dictionary of 65,536": (lambda: _wide(1 << 18, 16, np.int32), zf.ZF_DICT_BP, 1 << 18),
    "delta, narrow": (lambda: W.sorted_keys(3, 100_003), zf.ZF_DELTA_BP, 16384),
    "delta, 20 bits": (lambda: np.cumsum(_wide(30_000, 20, np.int64)), zf.ZF_DELTA_BP, 8192),
    "delta, 60 bits": (lambda: _wide(9_000, 60, np.int64), zf.ZF_DELTA_BP, 4096),
    "delta, int32 extremes": (lambda: np.tile(np.array([-2**31, 2**31 - 1, 0], np.int32), 3000), zf.ZF_DELTA_BP, 4096),
    "runs": (lambda: W.dates_rle(5, 50_001).astype(np.int64), zf.ZF_RLE, 7168),
    "runs of one": (lambda: np.arange(5000, dtype=np.int32), zf.ZF_RLE, 2048),
    "one run": (lambda: np.full(300_000, 9, np.int32), zf.ZF_RLE, 1 << 18),
    "raw": (lambda: _wide(10_007, 64, np.int64), zf.ZF_RAW, 4096),
    "prices of five jobs per chunk": (lambda: W.decimal_prices(1, 7, 0, 5_000_011), zf.ZF_FLOAT2INT, 17 * 1024),
    "full grid, four tiles a job": (lambda: _wide(20_000_003, 3, np.int32), zf.ZF_FOR_BP, 1 << 20),
}


def _call(col: bytes, out_bytes: int):
    import torch
    d = torch.frombuffer(bytearray(col), dtype=torch.uint8).cuda()
    out = torch.full((out_bytes + 64,), SENTINEL, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    st = zf.zf_decompress_device_noalloc(d.data_ptr(), d.numel(), out.data_ptr(), out_bytes)
    return st, out.cpu().numpy()


@pytest.mark.parametrize("name", COLUMNS)
def test_columns(name):
    make, scheme, chunk_rows = COLUMNS[name]
    x = make()
    h = compress(x, scheme, chunk_rows)
    col = zf.zf_compressed_bytes(h)
    zf.zf_compressed_free(h)
    st, out = _call(col, x.nbytes)
    assert st == zf.ZF_OK
    assert np.array_equal(out[:x.nbytes], x.view(np.uint8))
    assert (out[x.nbytes:] == SENTINEL).all()


def _set(fmt, pos, value):
    return lambda b: struct.pack_into(fmt, b, pos, value)


def test_malformed_columns_are_refused_and_the_next_call_works():
    x = W.sorted_keys(9, 40_000)
    h = compress(x, zf.ZF_DELTA_BP, 8192)
    col = zf.zf_compressed_bytes(h)
    zf.zf_compressed_free(h)
    c1, = struct.unpack_from("<Q", col, 64 + 32)                  # chunk 1
    entries = c1 + struct.unpack_from("<I", col, c1 + 24)[0]
    payload, = struct.unpack_from("<I", col, c1 + 40)
    for change, want in [
        (_set("<I", 0, 0), zf.ZF_ECORRUPT), (_set("<H", 4, 2), zf.ZF_ECORRUPT),
        (_set("<B", 7, zf.ZF_BYTES), zf.ZF_EUNSUPPORTED), (_set("<B", 6, zf.ZF_ANS), zf.ZF_EUNSUPPORTED),
        (_set("<B", 6, zf.ZF_LZ77), zf.ZF_ECORRUPT), (_set("<I", 8, 4097), zf.ZF_EINVAL),
        (_set("<I", 8, 4), zf.ZF_ECORRUPT), (_set("<I", 12, 1000), zf.ZF_ECORRUPT),
        (_set("<Q", 16, 1 << 40), zf.ZF_ECORRUPT), (_set("<Q", 32, len(col) + 16), zf.ZF_ECORRUPT),
        (_set("<Q", 64 + 32, c1 + 16), zf.ZF_ECORRUPT),            # chunk 1 does not follow chunk 0
        (_set("<Q", 64 + 40, 1 << 50), zf.ZF_ECORRUPT),            # its blob leaves the column
        (_set("<I", 64 + 56, 8191), zf.ZF_ECORRUPT),               # its directory rows
        (_set("<I", c1, 0), zf.ZF_ECORRUPT), (_set("<B", c1 + 4, zf.ZF_RLE), zf.ZF_ECORRUPT),
        (_set("<I", c1 + 8, 8191), zf.ZF_ECORRUPT), (_set("<I", c1 + 12, 9), zf.ZF_ECORRUPT),
        (_set("<I", c1 + 28, 1 << 30), zf.ZF_ECORRUPT),            # a section outside the blob
        (_set("<B", entries + 24 * 3 + 20, 65), zf.ZF_ECORRUPT),   # a block wider than the type
        (_set("<I", entries + 24 * 3 + 16, payload), zf.ZF_ECORRUPT),   # a payload past its section
        (_set("<I", entries + 24 * 3 + 16, 8), zf.ZF_ECORRUPT),    # a payload off its boundary
    ]:
        bad = bytearray(col)
        change(bad)
        st, out = _call(bytes(bad), x.nbytes)
        assert st == want
        assert (out[x.nbytes:] == SENTINEL).all()
        st, out = _call(col, x.nbytes)
        assert st == zf.ZF_OK and np.array_equal(out[:x.nbytes], x.view(np.uint8))
    assert _call(col, x.nbytes - 8)[0] == zf.ZF_EINVAL
    assert _call(col[:-16], x.nbytes)[0] == zf.ZF_ECORRUPT


def test_warps_of_several_jobs_and_a_malformed_late_chunk():
    """25M rows are 6,104 jobs of four tiles, more than one for the 4,864 warps
    of a full grid on 152 SMs: a warp's second job takes its descriptor's place
    while the first one's exceptions are patched, and in the malformed column
    without any check that joins the warp before."""
    n = 25_000_003
    x = np.round(np.random.default_rng(6).integers(0, 1 << 20, n) / 100.0, 2)
    x[::911] = np.nan                                              # exceptions all over the chunk
    h = compress(x, zf.ZF_FLOAT2INT, 8192)
    col = zf.zf_compressed_bytes(h)
    zf.zf_compressed_free(h)
    bad = bytearray(col)
    last, = struct.unpack_from("<Q", col, 64 + 32 * (n // 8192))   # the last chunk's blob
    struct.pack_into("<I", bad, last + 8, 1)                       # its rows
    for _ in range(3):
        st, out = _call(col, x.nbytes)
        assert st == zf.ZF_OK and np.array_equal(out[:x.nbytes], x.view(np.uint8))
        st, out = _call(bytes(bad), x.nbytes)
        assert st == zf.ZF_ECORRUPT and (out[x.nbytes:] == SENTINEL).all()


def test_overlapping_calls_get_their_own_answers():
    """Eight host threads call at once on streams of their own, half of them
    with a malformed column; every call gets its own answer, and so does every
    call after them."""
    import threading

    import torch
    x = np.arange(200_000, dtype=np.int64) * 3
    h = compress(x, zf.ZF_DELTA_BP, 8192)
    good = zf.zf_compressed_bytes(h)
    zf.zf_compressed_free(h)
    bad = bytearray(good)
    c5, = struct.unpack_from("<Q", good, 64 + 32 * 5)
    struct.pack_into("<I", bad, c5 + 8, 1)
    wrong = []

    def worker(i):
        stream = torch.cuda.Stream()
        col = torch.frombuffer(bytearray(bad if i % 2 else good), dtype=torch.uint8).cuda()
        out = torch.zeros(x.nbytes, dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        start.wait()
        for _ in range(200):
            st = zf.zf_decompress_device_noalloc(col.data_ptr(), col.numel(), out.data_ptr(), x.nbytes, stream.cuda_stream)
            if st != (zf.ZF_ECORRUPT if i % 2 else zf.ZF_OK):
                wrong.append((i, st))
        if i % 2 == 0 and not np.array_equal(out.cpu().numpy(), x.view(np.uint8)):
            wrong.append((i, "output"))

    start = threading.Barrier(8)
    threads = [threading.Thread(target=worker, args=(i,)) for i in range(8)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong
    for _ in range(70):                                            # more calls than result words
        assert _call(bytes(bad), x.nbytes)[0] == zf.ZF_ECORRUPT
        assert _call(good, x.nbytes)[0] == zf.ZF_OK


@pytest.mark.parametrize("scheme", ["for", "dict", "delta", "rle", "float2int", "raw"])
@pytest.mark.parametrize("where", ["header", "sections"])
def test_nothing_is_decoded_of_a_malformed_column(scheme, where):
    """A fault in the last of many chunks leaves the whole output as it was."""
    n = 70 * 8192 + 5
    make = {"for": (lambda: _wide(n, 17, np.int32), zf.ZF_FOR_BP), "dict": (lambda: _wide(n, 6, np.int64), zf.ZF_DICT_BP),
            "delta": (lambda: W.sorted_keys(4, n), zf.ZF_DELTA_BP), "rle": (lambda: W.dates_rle(4, n), zf.ZF_RLE),
            "float2int": (lambda: np.where(np.arange(n) % 5 == 0, np.nan, W.decimal_prices(1, 7, 0, n)), zf.ZF_FLOAT2INT),
            "raw": (lambda: _wide(n, 64, np.int64), zf.ZF_RAW)}[scheme]
    x = make[0]()
    h = compress(x, make[1], 8192)
    col = zf.zf_compressed_bytes(h)
    zf.zf_compressed_free(h)
    bad = bytearray(col)
    blob, = struct.unpack_from("<Q", col, 64 + 32 * 70)            # the last chunk, 5 rows
    off = struct.unpack_from("<III", col, blob + 24)
    if where == "header":
        struct.pack_into("<I", bad, blob, 0)
    elif scheme == "delta":
        struct.pack_into("<B", bad, blob + off[0] + 20, 65)        # a block wider than the type
    elif scheme == "float2int":
        struct.pack_into("<I", bad, blob + off[1], 5)              # an exception past the chunk
    else:
        length, = struct.unpack_from("<I", col, blob + 36)
        struct.pack_into("<I", bad, blob + 36, length + 4)         # the first section's length
    st, out = _call(bytes(bad), x.nbytes)
    assert st == zf.ZF_ECORRUPT and (out == SENTINEL).all()
    st, out = _call(col, x.nbytes)
    assert st == zf.ZF_OK and np.array_equal(out[:x.nbytes], x.view(np.uint8))
