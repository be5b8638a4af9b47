"""Rows of A cut into chunks (C of at most 1024 columns, more than 256 A
entries): lengths around the 256-entry chunk and the steps of its warps, rows
shared by several blocks, columns that no product reaches, empty rows of B."""

import numpy as np
import pytest

from oracle import OMat
from parity import assert_matches, oracle_product
from workloads import CSR, MIN_PLUS_I32, PLUS_TIMES_F64, random_batch

pytestmark = pytest.mark.gpu

LENGTHS = [1, 64, 255, 256, 257, 258, 511, 512, 513, 767, 768, 769, 1023, 1024, 1025, 2049, 5000, 20000]


@pytest.mark.parametrize("sr", [PLUS_TIMES_F64, MIN_PLUS_I32])
@pytest.mark.parametrize("m", [1, 31, 33, 256, 1024])
def test_split_rows_at_chunk_edges(dspg, m, sr):
    rng = np.random.default_rng(m + sr)
    k = 20011

    def csr(rows, ncols):
        rp = np.zeros(len(rows) + 1, np.int64)
        np.cumsum([len(r) for r in rows], out=rp[1:])
        col = np.concatenate([np.sort(r) for r in rows]).astype(np.int32)
        val = rng.random(col.shape[0]) - 0.5 if sr == PLUS_TIMES_F64 else rng.integers(-50, 51, col.shape[0], dtype=np.int32)
        return CSR(len(rows), ncols, rp, col, val)

    blen = rng.integers(0, min(m, 6) + 1, k)
    blen[:40] = min(m, 300)  # a few long rows of B among the empty and short ones
    B = csr([rng.choice(m, size=int(b), replace=False) for b in blen], m)
    A = csr([rng.choice(k, size=n, replace=False) for n in LENGTHS for _ in range(3)], k)
    g = dspg.DynamicSpGEMM(A, B)
    Ao, Bo = OMat.from_csr(A), OMat.from_csr(B)
    assert_matches(g.read_C(), *oracle_product(Ao, Bo), what="static")
    for t in range(3):
        b = random_batch(A.nrows, k, 200, 7 + t, sr, A=Ao.to_csr())
        g.apply_batch(b)
        Ao.apply(b)
        assert_matches(g.read_C(), *oracle_product(Ao, Bo), what=f"batch {t}")
    g.close()
