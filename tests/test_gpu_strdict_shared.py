"""String-dictionary decode around the sizes where the shared-memory kernel's
batches (64 tokens), tiles (1024 tokens), dictionaries and CTA ranges begin and
end, columns whose chunks take both kernels (dictionaries that fit in shared
memory and ones that do not), and short chunks on either side of the four per
SM (608 on 152 SMs) from which a call reads them through L1."""
import numpy as np
import pytest

import zf_workloads as W
from gpu_helpers import Gpu, out_specs

zf = pytest.importorskip("paper_2602_08190_gb300")
pytestmark = pytest.mark.gpu


def _words(seed, count, lo, hi):
    """`count` words of lo..hi letters, each ending in a space."""
    r = np.random.default_rng(seed)
    return [bytes(r.integers(97, 123, r.integers(lo, hi + 1) - 1).astype(np.uint8)) + b" " for _ in range(count)]


def _text(seed, words, tokens):
    r = np.random.default_rng(seed)
    return np.frombuffer(b"".join(words[i] for i in r.integers(0, len(words), tokens)), np.uint8).copy()


CASES = {
    "one token": lambda: (_text(1, [b"abc "], 1), 65536),
    "one word, a dictionary of one": (lambda: (_text(2, [b"abcdefg "], 5000), 65536)),
    "63 tokens": lambda: (_text(3, _words(3, 20, 2, 9), 63), 65536),
    "64 tokens": lambda: (_text(4, _words(4, 20, 2, 9), 64), 65536),
    "65 tokens of 64 bytes": lambda: (_text(5, _words(5, 20, 64, 64), 65), 65536),
    "1,023 tokens": lambda: (_text(6, _words(6, 200, 1, 12), 1023), 65536),
    "1,024 tokens": lambda: (_text(7, _words(7, 200, 1, 12), 1024), 65536),
    "1,025 tokens": lambda: (_text(8, _words(8, 200, 1, 12), 1025), 65536),
    "every length": lambda: (_text(9, _words(9, 900, 1, 64), 30_000), 131072),
    "single bytes": lambda: (np.random.default_rng(10).integers(0, 256, 200_003).astype(np.uint8), 65536),
    "1,025 entries": lambda: (_text(11, _words(11, 1025, 6, 8), 40_000), 1 << 20),
    "few short chunks": lambda: (_text(17, _words(17, 900, 3, 12), 4_500_000), 65536),
    "many short chunks": lambda: (_text(18, _words(18, 900, 3, 12), 6_500_000), 65536),
    "chunks of one tile": lambda: (_text(19, _words(19, 500, 64, 64), 300_000), 65536),
    "CTA ranges across many chunks": lambda: (_text(12, _words(12, 3000, 3, 12), 900_000), 65536),
    "one chunk over all CTAs": lambda: (_text(13, _words(13, 5000, 3, 12), 500_000), 1 << 23),
    "dictionaries at the shared-memory limit": lambda: (_text(14, _words(14, 13_000, 6, 9), 300_000), 1 << 19),
    "both kernels": lambda: (np.concatenate([_text(15, _words(15, 40_000, 6, 12), 120_000), _text(16, _words(16, 50, 6, 12), 120_000)]), 1 << 19),
}


@pytest.mark.parametrize("name", CASES)
def test_columns(name):
    t, chunk = CASES[name]()
    r = np.random.default_rng(99)
    o = np.unique(np.concatenate([[0, len(t)], r.integers(0, len(t) + 1, 3)])).astype(np.int32)
    col = zf.Column(t, o)
    h = zf.zf_compress_host(zf.zf_plan(None, col, scheme=zf.ZF_STRDICT, chunk_rows=chunk), col)
    g = Gpu()
    try:
        for resident in (False, True):
            got_t, got_o = g.decode([h], out_specs(t, o), resident=resident)
            assert np.array_equal(got_t, t) and np.array_equal(got_o, o)
    finally:
        zf.zf_compressed_free(h)
        g.close()


# Warps that decode several tiles one after another reuse their window: each
# tile's last partial block has to be out before the next tile clears it.
# 16M tokens are 15,625 tiles, four for each of the 32 warps of 152 CTAs.
@pytest.mark.parametrize("lo,hi,tokens", [(1, 2, 20_000_000), (3, 4, 16_000_000)])
def test_warps_of_several_tiles(lo, hi, tokens):
    r = np.random.default_rng(lo)
    words = np.full((7, hi), ord(" "), np.uint8)
    lens = r.integers(lo, hi + 1, 7)
    for i, n in enumerate(lens):
        words[i, :n - 1] = 97 + i
    pick = r.integers(0, 7, tokens)
    t = words[pick].reshape(-1)[(np.arange(hi) < lens[pick][:, None]).reshape(-1)]
    o = np.array([0, len(t)], np.int32)
    col = zf.Column(t, o)
    h = zf.zf_compress_host(zf.zf_plan(None, col, scheme=zf.ZF_STRDICT, chunk_rows=1 << 26), col)
    g = Gpu()
    try:
        for _ in range(3):
            got_t, got_o = g.decode([h], out_specs(t, o), resident=True)
            assert np.array_equal(got_t, t) and np.array_equal(got_o, o)
    finally:
        zf.zf_compressed_free(h)
        g.close()


# Eight stages and more of few tiles each are decoded through L1, fewer or
# larger ones with the dictionary in shared memory.
@pytest.mark.parametrize("stage_mib", [1, 2, 64])
def test_stages(stage_mib):
    t, o = W.text_column(3, 48 << 20)
    col = zf.Column(t, o)
    h = zf.zf_compress_host(zf.zf_plan(None, col, scheme=zf.ZF_STRDICT, chunk_rows=1 << 20), col)
    g = Gpu(stage_bytes=stage_mib << 20)
    try:
        got_t, got_o = g.decode([h], out_specs(t, o))
        assert np.array_equal(got_t, t) and np.array_equal(got_o, o)
    finally:
        zf.zf_compressed_free(h)
        g.close()
