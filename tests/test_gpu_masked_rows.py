"""The masked merge where rows of C gain and lose entries in every proportion:
holes filled by new entries, by the row's last entries (past the new length
or not) or by both, rows past 2048 entries (read by a whole block) and rows
that outgrow their room; C' and its Bloom filter against the oracle."""

import numpy as np
import pytest

from oracle import OMat
from parity import assert_matches, oracle_product
from test_gpu_masked import _bloom_matches
from workloads import CSR, MIN_PLUS_I32, OP_DELETE, OP_INSERT, PLUS_TIMES_F64, Batch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sr", [PLUS_TIMES_F64, MIN_PLUS_I32])
def test_rows_that_gain_and_lose_entries(dspg, sr):
    rng = np.random.default_rng(17 + sr)
    m = 30000
    sizes = [1, 5, 31, 32, 33, 40, 64, 65, 100, 700, 3000, 9000]
    k = len(sizes)
    bcols = [np.sort(rng.choice(m, size=s, replace=False)) for s in sizes]

    def value(n):
        return rng.random(n) if sr == PLUS_TIMES_F64 else rng.integers(1, 101, n, dtype=np.int32)

    rp = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    B = CSR(k, m, rp, np.concatenate(bcols).astype(np.int32), value(int(rp[-1])))
    n = 24
    present = rng.random((n, k)) < 0.5
    present[:, 0] = True
    r, c = np.nonzero(present)
    arp = np.concatenate([[0], np.cumsum(present.sum(1))]).astype(np.int64)
    A = CSR(n, k, arp, c.astype(np.int32), value(r.shape[0]))
    g = dspg.DynamicSpGEMM(A, B, bloom=True)
    Ao, Bo = OMat.from_csr(A), OMat.from_csr(B)
    longest = 0
    for t in range(5):
        flip = rng.random((n, k)) < 0.35  # each row drops some terms and takes others up
        r, c = np.nonzero(flip)
        op = np.where(present[r, c], OP_DELETE, OP_INSERT).astype(np.uint8)
        b = Batch(r.astype(np.int32), c.astype(np.int32), value(r.shape[0]), op)
        present ^= flip
        g.apply_batch(b)
        Ao.apply(b)
        C_o, S_o = oracle_product(Ao, Bo)
        longest = max(longest, int(np.diff(C_o.rowptr).max()))
        assert_matches(g.read_C(), C_o, S_o, what=f"batch {t}")
        _bloom_matches(g, Ao, Bo, f"batch {t}")
    assert longest > 2048
    g.close()
