"""Sweeps and products over a matrix with one full row and one full column: their
groups of four slices keep a width per slice."""
import copy

import numpy as np
import pytest
import scipy.sparse as sp

from oracle.pdhg import pdhg_solve
from oracle.scaling import rescale
from paper_2512_06715_gb300.instances import build_instance
from tests.conftest import instance_lp
from tests.parity_helpers import rel_err, returned_candidate

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2512_06715_gb300 import build
    build.build()


def _with_full_row_and_column(periods):
    """A budget over all variables that never binds and a variable fixed to zero in
    every row."""
    inst = copy.copy(build_instance(9, 13, 5, periods, seed=periods))
    K = sp.csr_matrix((inst.val, inst.col, inst.row_ptr), shape=(inst.m, inst.n))
    K = sp.vstack([K, sp.csr_matrix(-np.ones((1, inst.n)))])
    K = sp.hstack([K, sp.csr_matrix(np.full((inst.m + 1, 1), 0.5))]).tocsr()
    K.sort_indices()
    inst.row_ptr, inst.col, inst.val = K.indptr.astype(np.int64), K.indices.astype(np.int32), K.data
    inst.q = np.append(inst.q, -1e6)
    inst.c, inst.l, inst.u = np.append(inst.c, 1.0), np.append(inst.l, 0.0), np.append(inst.u, 0.0)
    inst.m, inst.n = K.shape
    return inst


@pytest.mark.parametrize("periods", [12, 40])
@pytest.mark.parametrize("variant,grid", [(-1, 0), (0, 3), (1, 4), (2, 3), (4, 2)])
def test_fixed_steps(periods, variant, grid):
    """64 constant-step attempts in FP64 equal the oracle's to 1e-10, as the other
    variant tests ask."""
    from paper_2512_06715_gb300.pdhg import Workspace, default_opts
    inst = _with_full_row_and_column(periods)
    lp = instance_lp(inst)
    slp, _, _ = rescale(lp)
    eta, omega = 0.9, np.linalg.norm(slp.c) / np.linalg.norm(slp.q)
    ws = Workspace.from_instance(inst, default_opts(fixed_eta=eta, fixed_omega=omega, max_iters=64, tol=1e-30,
                                                    kernel_variant=variant, kernel_grid=grid))
    x, y, r = ws.solve()
    ws.close()
    ref = pdhg_solve(lp, fixed=dict(eta=eta, omega=omega), stop_after=64)
    assert rel_err(x.cpu().numpy(), y.cpu().numpy(), returned_candidate(lp, ref, r)) <= 1e-10


@pytest.mark.parametrize("precision,tol", [(0, 1e-14), (1, 1e-6)])
def test_products(precision, tol):
    """K~ v and K~^T v: each entry within the rounding of its sum of |K~_ij v_j|, whose
    error bound is (entries of the row) x 2^-53 (2^-24 for FP32), taken here as
    64 such units: FMA chains of n terms stay well inside sqrt(n) x 4."""
    from paper_2512_06715_gb300.pdhg import Workspace
    inst = _with_full_row_and_column(40)
    ws = Workspace.from_instance(inst)
    ws.prepare()
    dr, dc = (d.cpu().numpy() for d in ws.scaling())
    K = sp.diags(dr) @ inst.scipy_csr() @ sp.diags(dc)
    rng = np.random.default_rng(0)
    for A, transpose in ((K, False), (K.T.tocsr(), True)):
        v = rng.standard_normal(A.shape[1])
        got = ws.apply_K(torch.as_tensor(v), transpose=transpose, precision=precision).cpu().numpy()
        assert (np.abs(got - A @ v) <= 64 * tol * (abs(A) @ np.abs(v) + 1e-300)).all()
    ws.close()


def test_products_of_many_short_rows_and_a_longer_one():
    """1.4 million rows of three entries and one of 60: a group with a width per slice in
    a matrix too large for its widest slice to matter."""
    from paper_2512_06715_gb300.pdhg import Workspace
    m, n, w = 1_400_000, 1_000_000, 60
    rng = np.random.default_rng(5)
    col = np.concatenate([np.sort(rng.choice(n, w, replace=False)),
                          (rng.integers(0, n - 3, m)[:, None] + np.arange(3)).ravel()]).astype(np.int32)
    row_ptr = np.concatenate([[0], w + 3 * np.arange(m + 1)]).astype(np.int64)
    val = rng.standard_normal(len(col))
    ws = Workspace(row_ptr, col, val, np.ones(n), np.zeros(n), np.ones(n), np.zeros(m + 1), 0)
    ws.prepare()
    dr, dc = (d.cpu().numpy() for d in ws.scaling())
    K = sp.diags(dr) @ sp.csr_matrix((val, col, row_ptr), shape=(m + 1, n)) @ sp.diags(dc)
    for precision, tol in ((0, 1e-14), (1, 1e-6)):
        for A, transpose in ((K, False), (K.T.tocsr(), True)):
            v = rng.standard_normal(A.shape[1])
            got = ws.apply_K(torch.as_tensor(v), transpose=transpose, precision=precision).cpu().numpy()
            assert (np.abs(got - A @ v) <= 64 * tol * (abs(A) @ np.abs(v) + 1e-300)).all()
    ws.close()
