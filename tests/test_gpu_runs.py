"""Sweeps over slices whose k-columns are partly runs and partly explicit indices,
and over rows longer than one load of run words (16 k-columns at two slices a
warp, 8 at four)."""
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


def _with_sums(inst, width):
    """The LP with a redundant row sum_{k < width} x_{j+k} <= a bound that never
    binds for every second j: sliding windows whose runs overlap and break."""
    inst = copy.copy(inst)
    K = sp.csr_matrix((inst.val, inst.col, inst.row_ptr), shape=(inst.m, inst.n))
    first = np.arange(0, inst.n - width + 1, 2)
    cols = (first[:, None] + np.arange(width)).ravel()
    rows = np.repeat(np.arange(len(first)), width)
    W = sp.csr_matrix((np.ones(len(cols)), (rows, cols)), shape=(len(first), inst.n))
    sign = -1.0  # rows are K x >= q
    K = sp.vstack([K, sign * W]).tocsr()
    K.sort_indices()
    inst.row_ptr, inst.col, inst.val = K.indptr.astype(np.int64), K.indices.astype(np.int32), K.data
    inst.q = np.concatenate([inst.q, np.full(len(first), -1e3 * width)])
    inst.m = K.shape[0]
    return inst


# windows of one load and of more: 8 and 9 (four slices), 16 and 17 (two), 33
@pytest.mark.parametrize("periods,width", [(24, 8), (24, 9), (40, 16), (40, 17), (96, 33)])
@pytest.mark.parametrize("variant,grid", [(1, 4), (2, 3), (4, 2)])
def test_mixed_runs_and_long_rows(periods, width, variant, grid):
    """64 constant-step attempts in FP64 equal the oracle's to 1e-10, as the other
    variant tests ask."""
    from paper_2512_06715_gb300.pdhg import Workspace, default_opts
    inst = _with_sums(build_instance(9, 13, 5, periods, seed=periods), width)
    lp = instance_lp(inst)
    slp, _, _ = rescale(lp)
    eta, omega = 0.9, np.linalg.norm(slp.c) / np.linalg.norm(slp.q)
    ws = Workspace.from_instance(inst, default_opts(fixed_eta=eta, fixed_omega=omega, max_iters=64, tol=1e-30,
                                                    kernel_variant=variant, kernel_grid=grid))
    x, y, r = ws.solve()
    ws.close()
    ref = pdhg_solve(lp, fixed=dict(eta=eta, omega=omega), stop_after=64)
    assert rel_err(x.cpu().numpy(), y.cpu().numpy(), returned_candidate(lp, ref, r)) <= 1e-10
