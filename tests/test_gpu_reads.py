"""Rows of C read in column order, at the lengths and widths where the read's
kernels change their way: 64 entries (a warp in registers, then a block with a
bitmap), the bitmap's 1024-column stretches and 262144-column windows, and C
wider than 2^22 columns (a sorting network, and the radix sort past 16384
entries)."""

import numpy as np
import pytest

from oracle import OMat
from parity import assert_rows_match
from workloads import CSR, MIN_PLUS_I32, OP_SET, PLUS_TIMES_F64, Batch

pytestmark = pytest.mark.gpu

# around the longest rows that go through the network instead of the bitmap's
# windows: 256 entries a window, at most 4096
NETWORK = [255, 256, 257, 511, 512, 513, 767, 768, 769, 1023, 1024, 1025, 4095, 4096, 4097]
LENGTHS = [0, 1, 31, 32, 33, 63, 64, 65, 66, 127, 128, 129, 511, 513, 1025, 2048, 16384, 16385, 20000]


def _csr(rows, ncols, sr, rng):
    rp = np.zeros(len(rows) + 1, np.int64)
    np.cumsum([len(r) for r in rows], out=rp[1:])
    col = np.concatenate([np.sort(r) for r in rows]).astype(np.int32) if rp[-1] else np.zeros(0, np.int32)
    val = rng.random(col.shape[0]) if sr == PLUS_TIMES_F64 else rng.integers(1, 101, col.shape[0], dtype=np.int32)
    return CSR(len(rows), ncols, rp, col, val)


@pytest.mark.parametrize("sr", [PLUS_TIMES_F64, MIN_PLUS_I32])
@pytest.mark.parametrize("m", [20480, (1 << 18), (1 << 18) + 1, 600001, (1 << 22) + 33])
def test_rows_in_order_at_every_width(dspg, m, sr):
    _rows_in_order(dspg, m, sr, LENGTHS)


@pytest.mark.parametrize("sr", [PLUS_TIMES_F64, MIN_PLUS_I32])
@pytest.mark.parametrize("m", [1 << 18, (1 << 18) + 1, 600001, 1 << 20, 1 << 22])
def test_rows_in_order_by_network_and_by_windows(dspg, m, sr):
    _rows_in_order(dspg, m, sr, NETWORK)


def _rows_in_order(dspg, m, sr, lengths):
    rng = np.random.default_rng(m + sr)
    edges = np.array([c for c in (0, 1, 1023, 1024, (1 << 18) - 1, 1 << 18, (1 << 18) + 1, m - 2, m - 1) if c < m])
    brows, arows = [], []
    for length in lengths:
        cols = np.unique(np.concatenate([edges[: max(0, length // 8)], rng.choice(m, size=length, replace=False)]))
        cols = rng.permutation(cols)[:length]
        # each row of C is the union of disjoint rows of B, so that its columns arrive in runs
        cut = np.array_split(cols, 3)
        arows.append(np.arange(len(brows), len(brows) + 3))
        brows += cut
    arows.append(np.array([len(brows)]))
    brows.append(rng.choice(m, size=5000, replace=False))  # one run: may leave its kernel in any order
    A, B = _csr(arows, len(brows), sr, rng), _csr(brows, m, sr, rng)
    g = dspg.DynamicSpGEMM(A, B)
    Ao, Bo = OMat.from_csr(A), OMat.from_csr(B)
    every = np.arange(A.nrows, dtype=np.int32)
    orp, ocol, oval = Ao.multiply_rows(Bo, every)
    sabs = Ao.multiply_rows(Bo, every, absval=True)[2] if sr == PLUS_TIMES_F64 else None
    C = g.read_C()
    assert_rows_match(C.rowptr, C.col, C.val, orp, ocol, oval, sabs, "host")
    rp, col, val = (x.cpu().numpy() for x in g.read_C_device())
    assert_rows_match(rp, col, val, orp, ocol, oval, sabs, "device")
    pick = rng.permutation(every)[:9]  # rows in any order
    orp, ocol, oval = Ao.multiply_rows(Bo, pick)
    sabs = Ao.multiply_rows(Bo, pick, absval=True)[2] if sr == PLUS_TIMES_F64 else None
    assert_rows_match(*g.read_rows_C(pick), orp, ocol, oval, sabs, "listed rows")
    first = A.rowptr[:-1]
    b = Batch(every, A.col[first], A.val[first] + A.val[first], np.full(every.size, OP_SET, np.uint8))
    g.apply_batch(b)
    Ao.apply(b)
    orp, ocol, oval = Ao.multiply_rows(Bo, every)
    sabs = Ao.multiply_rows(Bo, every, absval=True)[2] if sr == PLUS_TIMES_F64 else None
    rows, *got = g.read_affected()  # straight into page-locked arrays
    assert np.array_equal(rows, every)
    assert_rows_match(*got, orp, ocol, oval, sabs, "affected rows")
    g.close()


def test_fill_call_takes_the_row_pointers_of_its_count_call_only(dspg):
    """The fill call of a two-call read of all of C, or of listed rows, uses the
    row pointers of its count call; a batch, a read of the affected rows or of
    A in between makes it compute them again."""
    import ctypes
    sr = MIN_PLUS_I32
    rng = np.random.default_rng(3)
    rows = [rng.choice(300, size=int(rng.integers(0, 9)), replace=False) for _ in range(300)]
    A = _csr(rows, 300, sr, rng)
    g = dspg.DynamicSpGEMM(A)
    Ao = OMat.from_csr(A)
    lib, h = dspg.load(), g._h

    def batch(seed):
        from workloads import random_batch
        b = random_batch(300, 300, 40, seed, sr, A=Ao.to_csr())
        g.apply_batch(b)
        Ao.apply(b)

    def count(listed):
        nnz = ctypes.c_int64()
        if listed is None:
            assert lib.dspg_read_C(h, ctypes.byref(nnz), None, None, None, 0, None) == 0
        else:
            assert lib.dspg_read_rows_C(h, listed.ctypes.data, len(listed), ctypes.byref(nnz), None, None, None, 0, None) == 0
        return nnz

    def fill(listed, nnz):
        n = A.nrows if listed is None else len(listed)
        rp, col, val = np.zeros(n + 1, np.int64), np.zeros(100000, np.int32), np.zeros(100000, np.int32)
        out = (rp.ctypes.data, col.ctypes.data, val.ctypes.data, 0, None)
        if listed is None:
            assert lib.dspg_read_C(h, ctypes.byref(nnz), *out) == 0
        else:
            assert lib.dspg_read_rows_C(h, listed.ctypes.data, len(listed), ctypes.byref(nnz), *out) == 0
        every = np.arange(A.nrows, dtype=np.int32) if listed is None else listed
        assert_rows_match(rp, col[: rp[-1]], val[: rp[-1]], *Ao.multiply_rows(Ao, every), what="fill")

    some = rng.permutation(300)[:50].astype(np.int32)
    batch(1)
    for listed in (None, some):
        for between in (lambda: None, lambda: batch(2), lambda: g.read_affected(), lambda: g.read_A(),
                        lambda: count(some if listed is None else None)):
            nnz = count(listed)
            between()
            fill(listed, nnz)
            fill(listed, nnz)
    g.close()


@pytest.mark.parametrize("listed", [False, True])
def test_a_count_call_before_the_wait_does_not_serve_a_fill_after_it(dspg, listed):
    """The count call of a read made while an asynchronous batch is in flight
    (the batch's stream idle, so that nothing changes meanwhile): the fill call
    after the wait scans the lengths again, and when the wait has rerun the
    batch in larger arenas, returns C after that."""
    import ctypes
    import torch
    from workloads import random_batch, random_csr
    sr = MIN_PLUS_I32
    n = 400
    lib = dspg.load()
    some = np.random.default_rng(5).permutation(n)[:150].astype(np.int32)
    every = some if listed else np.arange(n, dtype=np.int32)

    def read(g, nnz, *out):
        if listed:
            assert lib.dspg_read_rows_C(g._h, some.ctypes.data, some.size, ctypes.byref(nnz), *out, 0, None) == 0
        else:
            assert lib.dspg_read_C(g._h, ctypes.byref(nnz), *out, 0, None) == 0

    for tight in (False, True):
        A = random_csr(n, n, 10, 31, sr)
        g = dspg.DynamicSpGEMM(A, **(dict(slack_min=0, slack_div=1 << 20, arena_headroom=1.0) if tight else {}))
        Ao = OMat.from_csr(A)
        nnz, grown = ctypes.c_int64(), 0
        rp, col, val = np.zeros(every.size + 1, np.int64), np.zeros(n * n, np.int32), np.zeros(n * n, np.int32)
        out = (rp.ctypes.data, col.ctypes.data, val.ctypes.data)

        def fill_launches():
            k = lib.dspg_kernel_launches()
            read(g, nnz, *out)
            k = lib.dspg_kernel_launches() - k
            assert_rows_match(rp, col[: rp[-1]], val[: rp[-1]], *Ao.multiply_rows(Ao, every), what=f"tight {tight}")
            return k

        for t in range(3):
            read(g, nnz, None, None, None)
            with_kept = fill_launches()
            b = random_batch(n, n, 3000 if tight else 60, 60 + t, sr, A=Ao.to_csr(), hit_frac=0.1)
            g.apply_batch_async(b)
            torch.cuda.synchronize()
            read(g, nnz, None, None, None)
            grown += g.apply_batch_wait()["compactions"]
            Ao.apply(b)
            assert fill_launches() > with_kept
        assert (grown > 0) == tight
        g.close()


@pytest.mark.parametrize("nr", [1, 3, 1023, 1025, 4095, 4096, 4097, 9000])
def test_affected_rows_around_the_one_block_read(dspg, nr):
    """R and its row pointers come from one block up to 4096 rows and from many
    beyond: both one-call reads, with R spread over the bitmap's chunks."""
    import torch
    rng = np.random.default_rng(nr)
    n, k, m = 30000, 150, 40
    A = _csr([rng.choice(k, size=int(rng.integers(0, 4)), replace=False) for _ in range(n)], k, MIN_PLUS_I32, rng)
    B = _csr([rng.choice(m, size=int(rng.integers(0, 6)), replace=False) for _ in range(k)], m, MIN_PLUS_I32, rng)
    g, g2 = dspg.DynamicSpGEMM(A, B), dspg.DynamicSpGEMM(A, B)
    Ao, Bo = OMat.from_csr(A), OMat.from_csr(B)
    for room in (nr, nr + 300):  # the arrays' room bounds what the launch is sized for
        rows = np.sort(rng.choice(n, size=nr, replace=False)).astype(np.int32)
        b = Batch(rng.permutation(rows), rng.integers(0, k, nr).astype(np.int32), rng.integers(1, 99, nr).astype(np.int32),
                  np.full(nr, OP_SET, np.uint8))
        out = (torch.empty(room, dtype=torch.int32, pin_memory=True).numpy(),
               torch.empty(room + 1, dtype=torch.int64, pin_memory=True).numpy(),
               torch.empty(room * 40 + 1, dtype=torch.int32, pin_memory=True).numpy(),
               torch.empty(room * 40 + 1, dtype=torch.int32, pin_memory=True).numpy())
        _, one = g.apply_read_affected(b, out=out)
        g2.apply_batch(b)
        two = g2.read_affected()
        Ao.apply(b)
        want = Ao.multiply_rows(Bo, rows)
        for got in (one, two):
            assert np.array_equal(got[0], rows)
            assert_rows_match(*got[1:], *want, what=f"{nr} rows")
    g.close()
    g2.close()


def test_whole_read_while_an_asynchronous_batch_rewrites_rows(dspg):
    """A read of all of C while a batch runs: the rows the batch cannot change
    come out whole, whatever the others hold, and the next read is right.  The
    rows of C have no slack, so that rows of more than 64 entries move to the
    arena's tail, in memory that held other values before."""
    import torch
    from workloads import random_batch
    sr = MIN_PLUS_I32
    rng = np.random.default_rng(12)
    n, m = 1500, 300000
    A = _csr([rng.choice(n, size=int(rng.integers(0, 30)), replace=False) for _ in range(n)], n, sr, rng)
    B = _csr([rng.choice(m, size=int(rng.integers(0, 200)), replace=False) for _ in range(n)], m, sr, rng)
    torch.cuda.empty_cache()
    junk = torch.randint(-2**31, 2**31 - 1, (1 << 28,), dtype=torch.int32, device="cuda")  # 1 GiB, given back
    torch.cuda.synchronize()
    del junk
    torch.cuda.empty_cache()
    g = dspg.DynamicSpGEMM(A, B, slack_min=0, slack_div=1 << 20, arena_headroom=6.0)
    Ao, Bo = OMat.from_csr(A), OMat.from_csr(B)
    every = np.arange(n, dtype=np.int32)
    side = torch.cuda.Stream()
    room_a = (np.diff(A.rowptr) + 3) // 4 * 4
    for t in range(6):
        b = random_batch(n, n, 400, 20 + t, sr, A=Ao.to_csr())
        g.apply_batch_async(b)
        mid = g.read_C(stream=side)
        st = g.apply_batch_wait()
        changed = np.zeros(n, bool)
        changed[g.last_affected()] = True
        orp, ocol, oval = Ao.multiply_rows(Bo, every)  # before the batch
        for i in np.nonzero(~changed)[0]:
            lo, hi = mid.rowptr[i], mid.rowptr[i + 1]
            assert np.array_equal(mid.col[lo:hi], ocol[orp[i]:orp[i + 1]]), f"batch {t}: row {i}"
            assert np.array_equal(mid.val[lo:hi], oval[orp[i]:orp[i + 1]]), f"batch {t}: row {i}"
        Ao.apply(b)
        C = g.read_C()
        want = Ao.multiply_rows(Bo, every)
        assert_rows_match(C.rowptr, C.col, C.val, *want, what=f"batch {t}")
        # of the rows that moved, those that are not A's and not short ones of C that grew are long rows of C
        len_a = np.diff(Ao.to_csr().rowptr)
        moved_a = len_a > room_a
        room_a[moved_a] = (len_a[moved_a] + 3) // 4 * 4
        short = np.sum((np.diff(want[0]) > np.diff(orp)) & (np.diff(want[0]) <= 64))
        assert st["relocations"] > moved_a.sum() + short and st["compactions"] == 0
    g.close()


@pytest.mark.parametrize("form", [False, True])
@pytest.mark.parametrize("on_device", [0, 1])
def test_reads_without_columns_or_without_values(dspg, form, on_device):
    """col and val may be NULL in a fill call, in host and in device memory."""
    import ctypes
    import torch
    sr = PLUS_TIMES_F64
    rng = np.random.default_rng(8)
    n = 90
    A = _csr([rng.choice(n, size=int(rng.integers(0, 40)), replace=False) for _ in range(n)], n, sr, rng)
    g = dspg.DynamicSpGEMM(A, **(dict(alpha=2.0, beta=1.0, X=A) if form else {}))
    want = g.read_C()
    lib = dspg.load()
    dev = "cuda" if on_device else "cpu"
    for with_col, with_val in ((True, False), (False, True), (False, False)):
        rp = torch.zeros(n + 1, dtype=torch.int64, device=dev)
        col = torch.full((want.col.size,), -7, dtype=torch.int32, device=dev)
        val = torch.full((want.col.size,), -7.0, dtype=torch.float64, device=dev)
        nnz = ctypes.c_int64()
        assert lib.dspg_read_C(g._h, ctypes.byref(nnz), rp.data_ptr(), col.data_ptr() if with_col else None,
                               val.data_ptr() if with_val else None, on_device, None) == 0
        assert nnz.value == want.col.size and np.array_equal(rp.cpu().numpy(), want.rowptr)
        assert np.array_equal(col.cpu().numpy(), want.col if with_col else np.full(want.col.size, -7))
        assert np.array_equal(val.cpu().numpy(), want.val if with_val else np.full(want.col.size, -7.0))
    g.close()


@pytest.mark.parametrize("shift", [0, 2, 4])
def test_affected_rows_into_arrays_off_their_alignment(dspg, shift):
    """Page-locked result arrays that start `shift` bytes past an aligned
    address get the same rows (through scratch where their values would be
    misaligned), by both one-call reads."""
    import torch
    from workloads import random_batch
    sr = PLUS_TIMES_F64
    rng = np.random.default_rng(shift)
    n = 500
    A = _csr([rng.choice(n, size=int(rng.integers(0, 30)), replace=False) for _ in range(n)], n, sr, rng)
    g = dspg.DynamicSpGEMM(A)
    Ao = OMat.from_csr(A)

    def pinned(count, dtype):
        raw = torch.empty(count * np.dtype(dtype).itemsize + 64, dtype=torch.uint8, pin_memory=True).numpy()
        return raw[shift: shift + count * np.dtype(dtype).itemsize].view(dtype)

    out = (pinned(n, np.int32), pinned(n + 1, np.int64), pinned(n * n, np.int32), pinned(n * n, np.float64))
    for t in range(3):
        b = random_batch(n, n, 60, t, sr, A=Ao.to_csr())
        _, got = g.apply_read_affected(b, out=out)
        got = [x.copy() for x in got]
        Ao.apply(b)
        rows = g.last_affected()
        want = Ao.multiply_rows(Ao, rows)
        sabs = Ao.multiply_rows(Ao, rows, absval=True)[2]
        for r in (got, g.read_affected(out=out)):
            assert np.array_equal(r[0], rows)
            assert_rows_match(*r[1:], *want, sabs, f"shift {shift}, batch {t}")
    g.close()
