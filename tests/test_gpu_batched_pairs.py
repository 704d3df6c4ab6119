"""Batched sweeps where the two instances of a lane take part differently: odd and
partial batches of the 64-slot layout, and steps accepted in one and rejected in the
other."""
import numpy as np
import pytest

from oracle.lp import kkt, lp_from_arrays
from paper_2512_06715_gb300.instances import build_instance, node_fixings

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2512_06715_gb300 import build
    build.build()


@pytest.mark.parametrize("B", [1, 31, 33, 63, 64])
@pytest.mark.parametrize("attempts", [64, 320])
def test_reported_measures_match_the_oracle(B, attempts):
    """Adaptive attempts with rejected steps (the acceptance counts differ between the
    instances after 320): every instance's reported rel-KKT and objective equal the
    oracle's recomputation from its returned point -- to 1e-6 relative, the FP64 sums of
    a point that FP32 iterates made -- and untouched slots leave the others alone."""
    from paper_2512_06715_gb300.pdhg import Workspace, default_opts
    inst = build_instance(12, 18, 10, 12, seed=3, with_slack=True)
    l_b, u_b = node_fixings(inst, B)
    ws = Workspace.from_instance(inst, default_opts(precision="mixed", tol=1e-12, max_iters=attempts,
                                                    time_limit_s=60.0))
    x, y, res = ws.solve_batched(l_b, u_b)
    ws.close()
    x, y = x.cpu().numpy(), y.cpu().numpy()
    if B > 1 and attempts == 320:
        assert len({r["accepted"] for r in res}) > 1
    for k, r in enumerate(res):
        lp = lp_from_arrays(inst.row_ptr, inst.col, inst.val, inst.q, inst.c, l_b[k], u_b[k], inst.m_eq)
        chk = kkt(lp, x[k], y[k])
        assert r["iterations"] == attempts
        assert abs(chk.rel_kkt - r["rel_kkt"]) <= 1e-6 * r["rel_kkt"], (k, chk.rel_kkt, r["rel_kkt"])
        assert abs(chk.primal_obj - r["primal_obj"]) <= 1e-6 * (1.0 + abs(chk.primal_obj))
