"""The sums and the waits that the blocks of the resident attempts share."""
import numpy as np
import pytest

from paper_2512_06715_gb300.instances import build_instance

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

COOPERATIVE = (500, 700, 60, 24)  # more blocks than a cluster has


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2512_06715_gb300 import build
    build.build()


@pytest.mark.parametrize("size", [(12, 18, 10, 12), (60, 90, 12, 24), COOPERATIVE])
@pytest.mark.parametrize("precision,rtol", [("fp64", 1e-8), ("mixed", 1e-3)])
def test_adaptive_steps(size, precision, rtol):
    """64 adaptive attempts: eta, the decision, eta_max (the ratio of the sums over all
    blocks of ||dx||^2, ||dy||^2 and dy^T K dx) and the next step of every attempt equal
    the separate kernels'.  The sums of both are in fixed but different orders; the
    tolerance is that of the adaptive replay for eta_max (FP64), and for FP32 sums of
    up to 1e5 terms 1e5 x 2^-24 of rounding at most in each.  A stale or a missing
    part of one block is off by about one part in the number of blocks or more."""
    from paper_2512_06715_gb300.pdhg import Workspace, default_opts
    inst = build_instance(*size, seed=1)
    got = []
    for kw in (dict(kernel_variant=1), {}):
        ws = Workspace.from_instance(inst, default_opts(precision=precision, max_iters=64, tol=1e-30, trace=1,
                                                        step_growth_exp=8.0, **kw))
        r = ws.solve()[2]
        got.append((ws.trace()[0], r["kernel_launches"]))
        ws.close()
    (one, n1), (res, n2) = got
    assert n2 < n1 and len(one) == len(res) == 64
    assert np.array_equal(one[:, 2], res[:, 2])
    for k in (0, 3, 4):
        fin = np.isfinite(one[:, k])
        assert np.array_equal(fin, np.isfinite(res[:, k]))
        assert np.allclose(one[fin, k], res[fin, k], rtol=rtol, atol=0), k


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("host_loop", [0, 1])
def test_a_wait_that_gives_up(precision, host_loop):
    """A limit of no polls ends the solve with TIMEOUT; with the default limit the same
    workspace then solves as if nothing had been."""
    from paper_2512_06715_gb300.pdhg import INJECT_WAIT_POLLS, PDHGError, Workspace, default_opts
    inst = build_instance(*COOPERATIVE, seed=1)
    ws = Workspace.from_instance(inst, default_opts(precision=precision, max_iters=128, tol=1e-30, host_loop=host_loop))
    x0, y0, r0 = ws.solve()
    ws.inject(INJECT_WAIT_POLLS, 0)
    for _ in range(2):
        with pytest.raises(PDHGError, match="TIMEOUT"):
            ws.solve()
    ws.inject(INJECT_WAIT_POLLS, -1)
    x, y, r = ws.solve()
    ws.close()
    assert r["kernel_launches"] == r0["kernel_launches"] and r["rel_kkt"] == r0["rel_kkt"]
    assert torch.equal(x, x0) and torch.equal(y, y0)
