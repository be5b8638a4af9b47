"""The hash kernels at every table size with products that never, at random or
always find their column there already (rows of B apart, overlapping by all
but one column, and the same), in the static product and after a batch: the
products of one round that share a column meet in its slot."""

import numpy as np
import pytest

from oracle import OMat
from parity import assert_matches, oracle_product
from workloads import CSR, MIN_PLUS_I32, PLUS_TIMES_F64, random_batch

pytestmark = pytest.mark.gpu


def _csr(cols, ncols, sr, rng):
    cols = np.sort(cols, 1).astype(np.int32)
    val = rng.random(cols.size) - 0.5 if sr == PLUS_TIMES_F64 else rng.integers(-50, 51, cols.size, dtype=np.int32)
    return CSR(cols.shape[0], ncols, np.arange(cols.shape[0] + 1, dtype=np.int64) * cols.shape[1], cols.reshape(-1), val)


@pytest.mark.parametrize("sr", [PLUS_TIMES_F64, MIN_PLUS_I32])
@pytest.mark.parametrize("kind", ["apart", "band", "same"])
@pytest.mark.parametrize("d", [9, 11, 15, 22, 31, 45, 64, 90, 127])  # d * d products a row: a table size each
def test_products_that_share_columns(dspg, d, kind, sr):
    rng = np.random.default_rng(d)
    rows, k, m = 70, 3 * d, 20011
    a = np.stack([rng.choice(k, d, replace=False) for _ in range(rows)])
    if kind == "apart":  # k * d <= 3 * 127 * 127 columns, folded into m
        b = np.stack([(i * 1009 + np.arange(d) * 31) % m for i in range(k)])
    elif kind == "band":
        b = np.arange(k)[:, None] + np.arange(d)[None]
    else:
        b = np.broadcast_to(np.arange(d) * 7, (k, d))
    A, B = _csr(a, k, sr, rng), _csr(b, m, sr, rng)
    g = dspg.DynamicSpGEMM(A, B)
    Ao, Bo = OMat.from_csr(A), OMat.from_csr(B)
    assert_matches(g.read_C(), *oracle_product(Ao, Bo), what="static")
    u = random_batch(rows, k, 200, d, sr, A=Ao.to_csr())
    g.apply_batch(u)
    Ao.apply(u)
    assert_matches(g.read_C(), *oracle_product(Ao, Bo), what="batch")
    g.close()
