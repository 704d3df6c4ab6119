"""A driver that refuses the launch of the resident attempts: the separate kernels take
over, timed like those of any other LP, and stay."""
import numpy as np
import pytest

from oracle.scaling import rescale
from paper_2512_06715_gb300.instances import build_instance
from tests.conftest import instance_lp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2512_06715_gb300 import build
    build.build()


@pytest.mark.parametrize("precision,per_check", [("fp64", 127), ("mixed", 128)])
@pytest.mark.parametrize("host_loop", [0, 1])
@pytest.mark.parametrize("solved_before", [False, True])
def test_refused(precision, per_check, host_loop, solved_before, monkeypatch, capfd):
    """128 constant-step attempts (two checks), refused at the first solve or after a
    resident one: the same point to 1e-10 (FP64; 1e-5 FP32), kernel_launches of the
    separate kernels then and ever after, their shapes timed by the second solve."""
    from paper_2512_06715_gb300.pdhg import INJECT_RESIDENT_REFUSED, Workspace, default_opts
    inst = build_instance(12, 18, 10, 12, seed=1)
    slp, _, _ = rescale(instance_lp(inst))
    opts = dict(precision=precision, max_iters=128, tol=1e-30, host_loop=host_loop, fixed_eta=0.9,
                fixed_omega=np.linalg.norm(slp.c) / np.linalg.norm(slp.q))
    ws = Workspace.from_instance(inst, default_opts(**opts))
    x0, y0, r0 = ws.solve()
    if not solved_before:
        ws.close()
        ws = Workspace.from_instance(inst, default_opts(**opts))
    monkeypatch.setenv("UCPDHG_TUNE_LOG", "1")
    ws.inject(INJECT_RESIDENT_REFUSED, 1)
    for k in range(4):
        if k == 2:
            ws.inject(INJECT_RESIDENT_REFUSED, 0)
        if k == 3:
            ws.set_opts(time_limit_s=100.0)
        x, y, r = ws.solve()
        assert r["iterations"] == 128 and r["kernel_launches"] == r0["kernel_launches"] + 2 * per_check
        for a, b in ((x, x0), (y, y0)):
            assert float((a - b).abs().max()) <= (1e-10 if precision == "fp64" else 1e-5) * float(b.abs().max())
        if k == 1:
            assert "dual variant" in capfd.readouterr().err
    ws.close()
