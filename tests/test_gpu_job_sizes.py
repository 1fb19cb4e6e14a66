"""Launches on either side of the row counts where the built-in job size of a
launch changes (rows per SM against 1,024- to 4,096-row jobs), for schemes that
are cut by different rules, alone and batched: every row is decoded once."""
import numpy as np
import pytest

from gpu_helpers import Gpu, compress, out_specs

zf = pytest.importorskip("paper_2602_08190_gb300")
pytestmark = pytest.mark.gpu

SMS = 152
ROWS = [4096 * 8 * SMS - 1, 4096 * 14 * SMS, 4096 * 20 * SMS + SMS, 4096 * 32 * SMS - 1]


def _column(name, n):
    r = np.random.default_rng(n)
    return {"for 24": lambda: (r.integers(0, 1 << 24, n).astype(np.int32), zf.ZF_FOR_BP),
            "for 40": lambda: (r.integers(0, 1 << 40, n), zf.ZF_FOR_BP),
            "dict": lambda: (r.integers(0, 1000, n), zf.ZF_DICT_BP),
            "delta": lambda: (np.cumsum(r.integers(0, 16, n)), zf.ZF_DELTA_BP)}[name]()


@pytest.mark.parametrize("name,chunk_rows", [("for 24", 65536), ("for 40", 1 << 20), ("dict", 65536), ("delta", 1 << 20)])
def test_job_sizes(name, chunk_rows):
    plain, batched = Gpu(), Gpu(flags=zf.ZF_KCFG_BATCHED)
    try:
        for n in ROWS:
            x, scheme = _column(name, n)
            h = compress(x, scheme, chunk_rows)
            for g in (plain, batched):
                got, = g.decode([h], out_specs(x), resident=True)
                assert np.array_equal(got, x)
            zf.zf_compressed_free(h)
    finally:
        plain.close()
        batched.close()
