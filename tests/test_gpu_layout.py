"""Sweeps over matrices whose slices mix the three ways their columns are found:
one run of consecutive columns, two runs, explicit indices."""
import numpy as np
import pytest

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


def _shuffled(inst, seed):
    """The same LP with its columns renumbered at random: no runs are left."""
    import copy
    import scipy.sparse as sp
    rng = np.random.default_rng(seed)
    perm = rng.permutation(inst.n)
    inst = copy.copy(inst)
    K = sp.csr_matrix((inst.val, inst.col, inst.row_ptr), shape=(inst.m, inst.n))[:, perm].tocsr()
    K.sort_indices()
    inst.row_ptr, inst.col, inst.val = K.indptr.astype(np.int64), K.indices.astype(np.int32), K.data
    inst.c, inst.l, inst.u = inst.c[perm], inst.l[perm], inst.u[perm]
    return inst


# periods: 32 and 96 are whole slices (one run), 48 and 33 straddle them (two runs),
# 7 leaves many short pieces (explicit indices); the last network has units alone
@pytest.mark.parametrize("periods", [7, 32, 33, 48, 96])
@pytest.mark.parametrize("shuffle", [False, True])
@pytest.mark.parametrize("variant,grid", [(1, 5), (2, 3), (4, 2), (0, 3)])
def test_fixed_steps_over_column_runs(periods, shuffle, variant, grid):
    """64 constant-step attempts in FP64 on few blocks (a warp sweeps groups of
    every kind and the ragged last one) equal the oracle's to 1e-10, as the other
    variant tests ask."""
    from paper_2512_06715_gb300.pdhg import Workspace, default_opts
    inst = build_instance(9, 13, 5, periods, seed=periods)
    if shuffle:
        inst = _shuffled(inst, periods)
    lp = instance_lp(inst)
    slp, _, _ = rescale(lp)
    eta, omega = 0.9, np.linalg.norm(slp.c) / np.linalg.norm(slp.q)
    ws = Workspace.from_instance(inst, default_opts(fixed_eta=eta, fixed_omega=omega, max_iters=64, tol=1e-30,
                                                    kernel_variant=variant, kernel_grid=grid))
    x, y, r = ws.solve()
    ws.close()
    ref = pdhg_solve(lp, fixed=dict(eta=eta, omega=omega), stop_after=64)
    assert rel_err(x.cpu().numpy(), y.cpu().numpy(), returned_candidate(lp, ref, r)) <= 1e-10
