"""Host batches: page-locked ones are read in place up to 16384 entries and
copied beyond, as pageable and misaligned ones always are."""

import numpy as np
import pytest

from oracle import OMat
from parity import assert_matches
from workloads import MIN_PLUS_I32, PLUS_TIMES_F64, Batch, random_batch, random_csr

pytestmark = pytest.mark.gpu


def _pinned(a, shift):
    """a in page-locked memory, its first byte `shift` past an aligned address."""
    import torch
    raw = torch.empty(a.nbytes + 64, dtype=torch.uint8, pin_memory=True).numpy()
    out = raw[shift: shift + a.nbytes].view(a.dtype) if a.nbytes else a
    out[...] = a
    return out


@pytest.mark.parametrize("sr", [PLUS_TIMES_F64, MIN_PLUS_I32])
@pytest.mark.parametrize("n", [1, 1000, 16384, 16385])
def test_page_locked_batches_in_place_and_copied(dspg, sr, n):
    A = random_csr(900, 700, 9, 3, sr)
    B = random_csr(700, 40, 5, 4, sr)
    handles = [dspg.DynamicSpGEMM(A, B) for _ in range(3)]
    Ao = OMat.from_csr(A)
    for t in range(3):
        b = random_batch(900, 700, n, 10 * n + t, sr, A=Ao.to_csr())
        kinds = [b] + [Batch(*(_pinned(x, s) for x in (b.row, b.col, b.val, b.op))) for s in (0, 2)]
        for g, k in zip(handles, kinds):
            g.apply_batch(k)
        Ao.apply(b)
        want = Ao.to_csr()
        for g, what in zip(handles, ("pageable", "page-locked", "misaligned")):
            assert_matches(g.read_A(), want, want, what=f"{what}, batch {t}")
    for g in handles:
        g.close()
