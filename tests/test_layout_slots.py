"""Padding of the internal layout, on the host: rows far longer than their neighbours."""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_2512_06715_gb300.instances import build_instance
from paper_2512_06715_gb300.pdhg import layout_slots


def _by_slices(lengths, first_eq):
    """Slots of 32-row slices of rows by decreasing length, equalities before inequalities."""
    order = np.concatenate([np.sort(lengths[:first_eq])[::-1], np.sort(lengths[first_eq:])[::-1]])
    order = np.concatenate([order, np.zeros(-len(order) % 32, order.dtype)])
    return 32 * int(order.reshape(-1, 32).max(axis=1).sum())


def _slots(K, m_eq):
    K = K.tocsr()
    K.sort_indices()
    k, kt = layout_slots(K.indptr, K.indices, K.data, K.shape[1], m_eq)
    per_row, per_col = np.diff(K.indptr), np.bincount(K.indices, minlength=K.shape[1])
    return (k, _by_slices(per_row, m_eq)), (kt, _by_slices(per_col, 0))


@pytest.mark.parametrize("dense", [1, 3])
@pytest.mark.parametrize("transposed", [False, True])
def test_long_rows_pad_their_slice_only(dense, transposed):
    """Sparse rows and `dense` full ones (budget rows), and the transpose (a variable in
    every row).  A group of four slices adds at most a quarter of its slots, or 128
    k-columns (4096 slots); beyond one group for the equalities and one for the
    inequalities the lengths are those of the sparse rows, of which none exceeds 42."""
    n = 40000
    rng = np.random.default_rng(dense)
    K = sp.random(3000, n, density=2e-4, random_state=rng, format="csr") + sp.csr_matrix(
        (np.ones(3000), (np.arange(3000), rng.integers(0, n, 3000))), shape=(3000, n))
    K = sp.vstack([K, sp.csr_matrix(np.ones((dense, n)))])
    for slots, alone in _slots(K.T if transposed else K, 0 if transposed else 1000):
        assert slots <= 1.25 * alone + 2 * 4096


@pytest.mark.parametrize("periods", [12, 48, 96])
def test_unit_commitment_rows_stay_in_groups(periods):
    """The layouts of the scheduling LPs are padded by a few per cent only."""
    inst = build_instance(60, 90, 12, periods, seed=1)
    K = inst.scipy_csr()
    for slots, alone in _slots(K, inst.m_eq):
        assert slots <= 1.25 * alone + 2 * 4096


def test_a_row_of_17_million_entries():
    """32 rows of it are 544 million slots: accepted, although 128 would exceed 2^31."""
    n = 17_000_000
    row_ptr = np.array([0, n, n + 2, n + 4], np.int64)
    col = np.concatenate([np.arange(n, dtype=np.int32), np.array([3, 5, 3, 7], np.int32)])
    k, _ = layout_slots(row_ptr, col, np.ones(n + 4), n, 0)
    assert k <= 32 * n + 4096


def test_a_failed_host_allocation_is_an_error_code():
    """In a process whose address space is nearly used up: an exception must not leave
    the C entry."""
    import subprocess
    import sys
    code = """
import resource
import numpy as np
from paper_2512_06715_gb300.pdhg import PDHGError, layout_slots
n = 4_000_000
row_ptr, col, val = np.array([0, n], np.int64), np.arange(n, dtype=np.int32), np.ones(n)
layout_slots(row_ptr[:1].repeat(2), col, val, n, 0)  # loads the library
used = int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()
resource.setrlimit(resource.RLIMIT_AS, (used + (60 << 20),) * 2)
try:
    layout_slots(row_ptr, col, val, n, 0)
except PDHGError as e:
    assert "NOMEM" in str(e), e
else:
    raise SystemExit("no error")
"""
    assert subprocess.run([sys.executable, "-c", code], timeout=120).returncode == 0
