"""Batches around the large sort's tiles (1024, 2048 and 4096 keys, one launch
per digit up to 2^20 entries) and its longer path: the last write of a key
wins, entry for entry, in batches that repeat keys many times."""

import numpy as np
import pytest

from workloads import CSR, MIN_PLUS_I32, OP_DELETE, Batch

pytestmark = pytest.mark.gpu

N, K = 1500, 1201


@pytest.mark.parametrize("n", [16385, 32768, 65536, 65537, 131073, 262144, 262145, 524289, 1048576, 1048577])
def test_last_write_wins_at_every_tile_size(dspg, n):
    rng = np.random.default_rng(n)
    empty = CSR(N, K, np.zeros(N + 1, np.int64), np.zeros(0, np.int32), np.zeros(0, np.int32))
    B = CSR(K, 4, np.arange(K + 1, dtype=np.int64), np.zeros(K, np.int32), np.ones(K, np.int32))
    g = dspg.DynamicSpGEMM(empty, B, semiring=MIN_PLUS_I32)
    state = {}
    for t in range(3):  # eager, captured, replayed
        m = n - t  # lengths of one launch size (but for the first of a power of two)
        skew = rng.random(m) < 0.3  # many keys share their leading digits
        row = np.where(skew, rng.integers(0, 3, m), rng.integers(0, N, m)).astype(np.int32)
        col = rng.integers(0, K, m).astype(np.int32)
        op = rng.integers(0, 3, m).astype(np.uint8)
        val = rng.integers(-1000, 1000, m, dtype=np.int32)
        g.apply_batch(Batch(row, col, val, op))
        key = row.astype(np.int64) * K + col
        order = np.argsort(key, kind="stable")
        last = order[np.append(key[order][1:] != key[order][:-1], True)]
        for k, o, v in zip(key[last].tolist(), op[last].tolist(), val[last].tolist()):
            if o == OP_DELETE:
                state.pop(k, None)
            else:
                state[k] = v
    keys = np.array(sorted(state), np.int64)
    A = g.read_A()
    assert np.array_equal(A.row_ids() * K + A.col, keys)
    assert np.array_equal(A.val, np.array([state[k] for k in keys.tolist()], np.int32))
    g.close()
