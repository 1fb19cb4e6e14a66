"""LZ77 blocks of hand-made tokens at the sizes where the decoders' batches
(512 and 32 tokens), lengths steps (2,048 bytes) and output segments (8,192
bytes) begin and end, against the oracle's decode of the same chunk: alone
(a CTA per block) and among 3,900 blocks of one launch (a warp per block)."""
import random
import struct

import numpy as np
import pytest

import oracle
from oracle_pins import _lz_blob

zf = pytest.importorskip("paper_2602_08190_gb300")
pytestmark = pytest.mark.gpu


def _varint(v: int, nbytes: int) -> bytes:
    return bytes([(v >> (7 * k)) & 0x7F | (0x80 if k + 1 < nbytes else 0) for k in range(nbytes)])


def _block(seed, tokens, lits, matches, offset, pad):
    """(blob, rows) of `tokens` tokens: literal and match lengths drawn from
    the given ranges, offsets from `offset(rng, position)`, every length padded
    to a drawn number of bytes when `pad`."""
    r = random.Random(seed)
    lengths, offs, lit, pos = b"", [], 0, 0
    for t in range(tokens):
        ll = r.randint(*lits)
        if pos == 0 and tokens > 1:
            ll = max(ll, 1)
        lengths += _varint(ll, max(r.randint(1, 3) if pad else 1, 1 if ll < 128 else 2 if ll < 1 << 14 else 3))
        pos += ll
        lit += ll
        if t + 1 < tokens:
            m = r.randint(*matches)
            lengths += _varint(m - 4, max(r.randint(1, 3) if pad else 1, 1 if m - 4 < 128 else 2 if m - 4 < 1 << 14 else 3))
            offs.append(min(pos, offset(r, pos)))
            pos += m
    assert pos <= 65536
    literals = bytes(r.randrange(256) for _ in range(lit))
    return _lz_blob(lengths, struct.pack(f"<{len(offs)}H", *offs), literals, pos, tokens), pos


def _column(blob: bytes, rows: int) -> bytes:
    total = 64 + 32 + len(blob)
    h = bytearray(64)
    struct.pack_into("<IHBBIIQQQI", h, 0, 0x4C4F435A, 1, zf.ZF_LZ77, zf.ZF_BYTES, 1, 65536, rows, rows, total, 0)
    return bytes(h) + struct.pack("<QQQII", 96, len(blob), 0, rows, 0) + blob


NEAR = lambda r, p: r.randint(1, 16)            # noqa: E731  chains through the bytes just written
FAR = lambda r, p: r.randint(1, min(p, 65535))  # noqa: E731
CASES = {
    "one literal": (1, (1, 1), (4, 4), NEAR, False),
    "literals alone, 65,535": (1, (65535, 65535), (4, 4), NEAR, False),
    "literals alone, 65,536": (1, (65536, 65536), (4, 4), NEAR, False),
    "two tokens, a run of one byte": (2, (0, 1), (65000, 65000), lambda r, p: 1, False),
    "two tokens, period 3": (2, (3, 5), (9000, 9000), lambda r, p: 3, False),
    "511 tokens": (511, (0, 3), (4, 20), FAR, False),
    "512 tokens": (512, (0, 3), (4, 20), NEAR, True),
    "513 tokens, the last one empty": (513, (0, 0), (4, 12), NEAR, False),
    "1,024 tokens, padded lengths": (1024, (0, 9), (4, 30), FAR, True),
    "1,025 tokens of 16 literals": (1025, (16, 16), (4, 40), FAR, False),
    "16,384 shortest tokens": (16384, (0, 0), (4, 4), NEAR, False),
    "long literal runs": (8, (7000, 8200), (4, 9), FAR, True),
    "512 tokens of 60 literals": (512, (60, 60), (4, 9), NEAR, False),
    "some 20 literals a token, padded": (1500, (10, 33), (4, 9), FAR, True),
    "some 150 literals a token": (300, (100, 205), (4, 20), FAR, False),
    "literal runs of a page and matches of one": (14, (2000, 2600), (2000, 2100), NEAR, False),
    "long matches": (12, (1, 2), (5000, 5400), FAR, False),
}


@pytest.mark.parametrize("name", CASES)
def test_hand_made_blocks(name):
    from gpu_helpers import Gpu
    g = Gpu()
    try:
        for seed in range(2):
            blob, rows = _block(seed, *CASES[name])
            want = oracle.default().decode_chunk(blob, np.uint8)
            h = zf.zf_compressed_from_bytes(_column(blob, rows))
            for resident in (False, True):
                got, = g.decode([h], [(np.uint8, rows)], resident=resident)
                assert np.array_equal(got, want)
            zf.zf_compressed_free(h)
    finally:
        g.close()


def test_hand_made_blocks_in_a_large_launch():
    import torch
    from gpu_helpers import Gpu
    blocks = [_block(seed, *CASES[name]) for name in CASES for seed in range(2)]
    want = [oracle.default().decode_chunk(b, np.uint8) for b, _ in blocks]
    handles = [zf.zf_compressed_from_bytes(_column(b, r)) for b, r in blocks]
    times = 150
    room = [(r + 127) // 128 * 128 for _, r in blocks]
    buf = torch.full((times * sum(room),), 0xA5, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    outs, caps, pos = [], [], 0
    for _ in range(times):
        for (_, r), n in zip(blocks, room):
            outs.append(buf.data_ptr() + pos)
            caps.append(r)
            pos += n
    g = Gpu()
    try:
        res = [zf.zf_upload(g.ctx, h) for h in handles]
        zf.zf_decompress_resident(g.ctx, res * times, outs, caps)
        zf.zf_sync(g.ctx)
        got = buf.cpu().numpy().reshape(times, -1)
        pos = 0
        for w, n in zip(want, room):
            assert np.array_equal(got[:, pos:pos + len(w)], np.broadcast_to(w, (times, len(w))))
            assert (got[:, pos + len(w):pos + n] == 0xA5).all()
            pos += n
        for r in res:
            zf.zf_resident_free(r)
    finally:
        g.close()
        for h in handles:
            zf.zf_compressed_free(h)


# Contents beyond text: a run that copies a run's end (its source lies in a
# match that overlaps its own output), runs after literals, periods, and
# blocks with more literals than a batch's ring, in launches of one block, of
# few and of many per SM.
def _runs(r, n):
    x = r.integers(0, 256, n).astype(np.uint8)
    x[(np.arange(n) // 512) % 2 == 0] = 0
    return x


def _padded(r, n):
    x = r.integers(0, 256, n).astype(np.uint8)
    x[(np.arange(n) % 100) < 60] = 32
    return x


CONTENTS = {
    "runs between literals": _runs,
    "padded fields": _padded,
    "long periods": lambda r, n: np.where(r.random(n) < 0.0003, r.integers(0, 256, n), np.resize(r.integers(0, 256, 37), n)).astype(np.uint8),
    "short runs": lambda r, n: np.repeat(r.integers(0, 3, n // 20 + 2), r.integers(1, 60, n // 20 + 2))[:n].astype(np.uint8),
    "zeros": lambda r, n: np.zeros(n, np.uint8),
}


@pytest.mark.parametrize("blocks", [1, 40, 1500, 2000])
@pytest.mark.parametrize("name", CONTENTS)
def test_contents(name, blocks):
    from gpu_helpers import Gpu
    n = blocks * 65536 - 77
    t = CONTENTS[name](np.random.default_rng(blocks), n)
    assert len(t) == n
    o = np.array([0, n], np.int32)
    col = zf.Column(t, o)
    h = zf.zf_compress_host(zf.zf_plan(None, col, scheme=zf.ZF_LZ77), col)
    g = Gpu()
    try:
        got, _ = g.decode([h], [(np.uint8, n), (np.int32, 2)], resident=True)
        assert np.array_equal(got, t)
    finally:
        zf.zf_compressed_free(h)
        g.close()
