"""The sizing pass: A rows around its steps of eight entries and its limits for
a thread, a warp and a block, with few rows (32 a block) and many (256 a block,
which hands out a bin's and C's places once a block)."""

import numpy as np
import pytest

from oracle import OMat
from parity import assert_matches, oracle_product
from workloads import CSR, MIN_PLUS_I32, PLUS_TIMES_F64, random_batch

pytestmark = pytest.mark.gpu

EDGES = [0, 1, 3, 4, 5, 7, 8, 9, 12, 15, 16, 17, 63, 64, 65, 511, 512, 513, 1500]


@pytest.mark.parametrize("sr", [PLUS_TIMES_F64, MIN_PLUS_I32])
@pytest.mark.parametrize("n", [1, 33, 257, 40003])
@pytest.mark.parametrize("m", [700, 6007])
def test_rows_of_every_step(dspg, n, m, sr):
    rng = np.random.default_rng(n + m + sr)
    k = 3001

    def csr(lens, ncols):
        rp = np.zeros(len(lens) + 1, np.int64)
        np.cumsum(lens, out=rp[1:])
        start = rng.integers(0, ncols, len(lens))
        step = np.repeat(start, lens) + np.arange(rp[-1]) - np.repeat(rp[:-1], lens)  # a run of columns per row
        row = np.repeat(np.arange(len(lens)), lens)
        col = step % ncols
        col = col[np.lexsort((col, row))].astype(np.int32)
        val = rng.random(col.shape[0]) - 0.5 if sr == PLUS_TIMES_F64 else rng.integers(-50, 51, col.shape[0], dtype=np.int32)
        return CSR(len(lens), ncols, rp, col, val)

    lens = rng.integers(0, 10, n)
    at = rng.permutation(n)[:4 * len(EDGES)]
    lens[at] = np.resize(EDGES, at.shape[0])
    A, B = csr(lens, k), csr(rng.integers(0, 5, k), m)
    g = dspg.DynamicSpGEMM(A, B)
    Ao, Bo = OMat.from_csr(A), OMat.from_csr(B)
    assert_matches(g.read_C(), *oracle_product(Ao, Bo), what="static")
    for t in range(2):
        b = random_batch(n, k, 2 * n, 11 + t, sr, A=Ao.to_csr())  # most rows change
        st = g.apply_batch(b)
        Ao.apply(b)
        assert st["a_entries"] <= Ao.to_csr().nnz
        assert_matches(g.read_C(), *oracle_product(Ao, Bo), what=f"batch {t}")
    g.close()
