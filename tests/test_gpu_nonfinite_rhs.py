"""A NaN or an infinity in the right-hand side of an inequality row that never has a
dual: the row's residual and its multiplier drop it (their clamps return the other
operand), so the check has to see it in q itself."""
import numpy as np
import pytest

from paper_2512_06715_gb300.instances import ROW_FLOW_NEG, ROW_FLOW_POS, build_instance, node_fixings

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2512_06715_gb300 import build
    build.build()


def _ws(value, **kw):
    """A day whose line limits are far from binding: no row of their slices has a dual.
    One of them gets `value`."""
    from paper_2512_06715_gb300.pdhg import Workspace, default_opts
    inst = build_instance(24, 38, 33, 24, seed=0, with_slack=True)
    lines = np.flatnonzero((inst.row_kind == ROW_FLOW_POS) | (inst.row_kind == ROW_FLOW_NEG))
    inst.q = inst.q.copy()
    inst.q[lines] -= 1e3
    inst.q[lines[len(lines) // 2]] = value
    return inst, Workspace.from_instance(inst, default_opts(max_iters=256, time_limit_s=60.0, **kw))


@pytest.mark.parametrize("value", [np.nan, -np.inf, np.inf])
@pytest.mark.parametrize("precision,variant", [("fp64", -1), ("fp64", 2), ("mixed", -1), ("mixed", 2)])
def test_single(value, precision, variant):
    """Resident and separate attempts: the first check reports it."""
    from paper_2512_06715_gb300.pdhg import PDHGError
    _, ws = _ws(value, precision=precision, kernel_variant=variant)
    with pytest.raises(PDHGError, match="NUMERIC"):
        ws.solve()
    ws.close()


@pytest.mark.parametrize("value", [np.nan, -np.inf, np.inf])
@pytest.mark.parametrize("B", [3, 40])
def test_batched(value, B):
    from paper_2512_06715_gb300.pdhg import PDHGError
    inst, ws = _ws(value, precision="mixed")
    with pytest.raises(PDHGError, match="NUMERIC"):
        ws.solve_batched(*node_fixings(inst, B))
    ws.close()
