"""The resident attempts (64 step attempts of a small LP in one launch) against the
oracle and against the separate per-attempt kernels.  (The adaptive schedule of a
resident run is replayed by test_gpu_pdhg.test_adaptive_schedule_replay.)"""
import numpy as np
import pytest

from oracle.pdhg import pdhg_solve
from oracle.scaling import rescale
from paper_2512_06715_gb300.instances import build_instance
from tests.conftest import instance_lp
from tests.parity_helpers import rel_err, returned_candidate

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# one block, clusters of 2 to 16 blocks with and without idle warps, and more
# blocks than a cluster has (a cooperative launch)
SIZES = [(1, 0, 1, 1), (4, 4, 4, 3), (12, 18, 10, 12), (24, 38, 33, 24), (60, 90, 12, 24), (500, 700, 60, 24)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2512_06715_gb300 import build
    build.build()


def _solve(inst, **kw):
    from paper_2512_06715_gb300.pdhg import Workspace, default_opts
    ws = Workspace.from_instance(inst, default_opts(tol=1e-30, time_limit_s=60.0, **kw))
    x, y, r = ws.solve()
    ws.close()
    return x.cpu().numpy(), y.cpu().numpy(), r


@pytest.mark.parametrize("size", SIZES)
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_fixed_steps(size, precision):
    """192 constant-step attempts: FP64 equals the oracle to 1e-10; FP32 equals the
    one-slice variant to 1e-5 (the same sums; FMA contraction may differ) and the
    oracle to 1e-4.  The launch count shows that the attempts ran resident."""
    N, L, G, T = size
    inst = build_instance(N, L, G, T, seed=1)
    lp = instance_lp(inst)
    slp, _, _ = rescale(lp)
    fixed = dict(eta=0.9 / max(1.0, np.abs(slp.K.data).max()), omega=max(np.linalg.norm(slp.c) / np.linalg.norm(slp.q), 1e-3))
    kw = dict(precision=precision, max_iters=192, fixed_eta=fixed["eta"], fixed_omega=fixed["omega"])
    x, y, r = _solve(inst, **kw)
    x1, y1, r1 = _solve(inst, kernel_variant=1, **kw)
    more = 127 if precision == "fp64" else 128  # FP32: the separate kernels flush the x window in a launch
    assert r["iterations"] == 192 and r["kernel_launches"] == r1["kernel_launches"] - 3 * more
    ref = pdhg_solve(lp, fixed=fixed, stop_after=192)
    err = rel_err(x, y, returned_candidate(lp, ref, r))
    assert err <= (1e-10 if precision == "fp64" else 1e-4), err
    assert np.abs(x - x1).max() <= 1e-5 * np.abs(x1).max() and np.abs(y - y1).max() <= 1e-5 * np.abs(y1).max()


def test_options_that_ask_for_the_separate_kernels():
    """A fixed variant, a fixed grid or launch overlap keeps the separate kernels,
    also after a resident solve of the same workspace, and back."""
    from paper_2512_06715_gb300.pdhg import Workspace, default_opts
    inst = build_instance(12, 18, 10, 12, seed=1)
    ws = Workspace.from_instance(inst, default_opts(max_iters=128, tol=1e-30))
    few = ws.solve()[2]["kernel_launches"]
    for kw in (dict(kernel_variant=2), dict(kernel_variant=-1, kernel_grid=2),
               dict(kernel_variant=-1, kernel_grid=0, launch_overlap=1)):
        ws.set_opts(**kw)
        r = ws.solve()[2]
        assert r["kernel_launches"] == few + 2 * 127 and r["launch_overlap"] == kw.get("launch_overlap", 0)
    ws.set_opts(launch_overlap=0)
    assert ws.solve()[2]["kernel_launches"] == few
    ws.close()
