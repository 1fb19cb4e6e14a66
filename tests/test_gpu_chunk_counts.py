"""Calls whose launches have about as many chunks as travel as kernel
parameters (64), one launch's descriptors or several launches' together, in
each way of running a call."""
import numpy as np
import pytest

from gpu_helpers import Gpu, compress, out_specs

zf = pytest.importorskip("paper_2602_08190_gb300")
pytestmark = pytest.mark.gpu

CHUNK = 4096
FLAGS = {"plain": 0, "batched": zf.ZF_KCFG_BATCHED, "graph": zf.ZF_KCFG_GRAPH,
         "batched graph": zf.ZF_KCFG_BATCHED | zf.ZF_KCFG_GRAPH}


def _column(scheme, chunks):
    """A column of `chunks` chunks, the last one of 7 rows (text: bytes)."""
    r = np.random.default_rng(chunks * 16 + scheme)
    if scheme in (zf.ZF_LZ77, zf.ZF_STRDICT):
        words = [bytes(r.integers(97, 123, k % 9 + 2).astype(np.uint8)) + b" " for k in range(200)]
        n = (chunks - 1) * 65536 + 7
        t = np.frombuffer(b"".join(words[i] for i in r.integers(0, 200, n // 3 + 8)), np.uint8)[:n].copy()
        o = np.array([0, n // 3, n], np.int32)
        col = zf.Column(t, o)
        return zf.zf_compress_host(zf.zf_plan(None, col, scheme=scheme, chunk_rows=65536), col), [t, o], out_specs(t, o)
    n = (chunks - 1) * CHUNK + 7
    x = {zf.ZF_FOR_BP: lambda: r.integers(-50, 900, n).astype(np.int32),
         zf.ZF_DICT_BP: lambda: r.integers(0, 20, n) * 1_000_003,
         zf.ZF_DELTA_BP: lambda: np.cumsum(r.integers(0, 9, n)),
         zf.ZF_RLE: lambda: np.repeat(r.integers(0, 99, n // 8 + 1), 8)[:n].astype(np.int32),
         zf.ZF_FLOAT2INT: lambda: r.integers(0, 10**6, n) / 100.0,
         zf.ZF_ANS: lambda: r.integers(0, 3, n).astype(np.int32)}[scheme]()
    return compress(x, scheme, CHUNK), [x], out_specs(x)


SCHEMES = [zf.ZF_FOR_BP, zf.ZF_DICT_BP, zf.ZF_DELTA_BP, zf.ZF_RLE, zf.ZF_FLOAT2INT, zf.ZF_ANS, zf.ZF_STRDICT, zf.ZF_LZ77]


@pytest.mark.parametrize("flags", FLAGS)
@pytest.mark.parametrize("counts", [(1,), (63,), (64,), (65,), (129,), (64, 1), (65, 1), (3, 66)])
def test_chunks_of_a_launch(flags, counts):
    g = Gpu(flags=FLAGS[flags], stage_bytes=1 << 30)    # one stage: a launch has all the chunks of its scheme
    try:
        for k, scheme in enumerate(SCHEMES):
            # further columns are of other schemes: launches of their own, or the same batched one
            cols = [_column(SCHEMES[(k + j) % len(SCHEMES)], n) for j, n in enumerate(counts)]
            want, specs = [x for c in cols for x in c[1]], [s for c in cols for s in c[2]]
            for resident in (False, True, False):       # with a graph: captured, then replayed
                got = g.decode([c[0] for c in cols], specs, resident=resident)
                for x, y in zip(got, want):
                    assert np.array_equal(x.view(np.uint8), np.ascontiguousarray(y).view(np.uint8))
            for c in cols:
                zf.zf_compressed_free(c[0])
    finally:
        g.close()
