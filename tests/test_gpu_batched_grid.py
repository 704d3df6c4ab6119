"""The batched sweeps' sums over the grid: groups of 16 blocks, then the groups."""
import numpy as np
import pytest

from paper_2512_06715_gb300.instances import build_instance, node_fixings

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2512_06715_gb300 import build
    build.build()


@pytest.mark.parametrize("B", [5, 64])
@pytest.mark.parametrize("grid", [15, 16, 17, 32, 33, 257])
def test_steps_do_not_depend_on_the_grid(B, grid):
    """Step sizes that soon stop growing (growth exponent 8: no step is rejected for a
    rounding error) after 64 attempts, and the points reached: those of one block to
    1e-4.  The grid changes the order of FP32 partial sums only, 1e-6 relative in a
    sum and a step; a stale or a missing sum is another step size from the first
    attempts on."""
    from paper_2512_06715_gb300.pdhg import Workspace, default_opts
    inst = build_instance(12, 18, 10, 12, seed=3, with_slack=True)
    l_b, u_b = node_fixings(inst, B)
    got = []
    for g in (1, grid):
        ws = Workspace.from_instance(inst, default_opts(precision="mixed", tol=1e-12, max_iters=64, autotune=0,
                                                        kernel_grid=g, step_growth_exp=8.0))
        x, y, res = ws.solve_batched(l_b, u_b)
        ws.close()
        assert all(r["iterations"] == 64 for r in res)
        got.append((np.array([r["eta"] for r in res]), x.cpu().numpy(), y.cpu().numpy()))
    for one, many in zip(*got):
        assert np.linalg.norm(many - one) <= 1e-4 * np.linalg.norm(one)
