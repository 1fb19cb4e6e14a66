"""RLE tiles around the run counts where a step of the presum ends (128 and 256
length entries, at each alignment of the tile's first run), with runs that
begin and end at tile and chunk borders, long runs over many tiles, and
malformed lengths."""
import struct

import numpy as np
import pytest

import oracle
from gpu_helpers import Gpu, compress, out_specs
from oracle_pins import chunks_of

zf = pytest.importorskip("paper_2602_08190_gb300")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    g = Gpu()
    yield g
    g.close()


def _check(gpu, x, chunk):
    h = compress(x, zf.ZF_RLE, chunk)
    try:
        for resident in (False, True):
            got, = gpu.decode([h], out_specs(x), resident=resident)
            assert np.array_equal(got, x)
    finally:
        zf.zf_compressed_free(h)


def _column(lengths, dt):
    v = np.arange(len(lengths)) % 7 * 1000 - 3
    return np.repeat(v, lengths).astype(dt)


@pytest.mark.parametrize("runs", [1, 2, 3, 124, 125, 126, 127, 128, 129, 130, 131, 132, 253, 254, 255, 256, 257, 258, 260, 512, 1023, 1024])
def test_runs_per_tile(gpu, runs):
    r = np.random.default_rng(runs)
    for shift in range(4):                              # the first run of a tile at each of four alignments
        parts = [np.ones(shift, int)] if shift else []
        for _ in range(6):
            cut = np.sort(r.choice(np.arange(1, 1024), runs - 1, replace=False)) if runs > 1 else np.array([], int)
            parts.append(np.diff(np.concatenate([[0], cut, [1024]])))
        lengths = np.concatenate(parts)
        for dt in (np.int32, np.int64):
            _check(gpu, _column(lengths, dt), 4096)


@pytest.mark.parametrize("lengths", [[1024] * 9, [1023, 1, 1024, 1025, 1, 2047, 2049], [5000, 1, 3, 9000, 2], [4096, 4096, 1],
                                     [1, 4095, 4097], [20000], [1, 20000, 1]])
def test_runs_across_tiles_and_chunks(gpu, lengths):
    for dt in (np.int32, np.int64):
        _check(gpu, _column(lengths, dt), 4096)


@pytest.mark.parametrize("value", [0, 2, 1 << 20, (1 << 31) - 1, 1 << 31, (1 << 32) - 1])
@pytest.mark.parametrize("run", [0, 1, 100, 127, 128, 300])
def test_malformed_lengths(gpu, run, value):
    """One length of a chunk of 3,072 rows in runs of eight replaced."""
    x = _column([8] * 384, np.int32)
    b = bytearray(oracle.encode(x, oracle.RLE, 4096))
    off, ln, r0, rows, ch = chunks_of(oracle.default(), bytes(b))[0]
    struct.pack_into("<I", b, off + ch["offs"][1] + 4 * run, value)
    h = zf.zf_compressed_from_bytes(bytes(b))
    gpu.decode([h], out_specs(x), expect=zf.ZF_ECORRUPT)
    zf.zf_compressed_free(h)
