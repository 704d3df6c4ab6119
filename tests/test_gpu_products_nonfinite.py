"""Products with an infinite or missing entry: the rows that have an entry in its column
show it, the others do not (their padding slots gather neighbouring columns)."""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_2512_06715_gb300.instances import build_instance

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2512_06715_gb300 import build
    build.build()


@pytest.mark.parametrize("periods", [7, 24, 33])
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_products(periods, value):
    """Every 7th column (row) in turn, both ways and in both precisions."""
    from paper_2512_06715_gb300.pdhg import Workspace
    inst = build_instance(9, 13, 5, periods, seed=periods)
    ws = Workspace.from_instance(inst)
    ws.prepare()
    dr, dc = (d.cpu().numpy() for d in ws.scaling())
    K = sp.diags(dr) @ inst.scipy_csr() @ sp.diags(dc)
    rng = np.random.default_rng(0)
    for A, transpose in ((K.tocsr(), False), (K.T.tocsr(), True)):
        v = torch.as_tensor(rng.standard_normal(A.shape[1]), device="cuda")
        for precision in (0, 1):
            plain = ws.apply_K(v, transpose=transpose, precision=precision).cpu().numpy()
            for j in range(0, A.shape[1], 7):
                w = v.clone()
                w[j] = value
                got = ws.apply_K(w, transpose=transpose, precision=precision).cpu().numpy()
                at = A[:, [j]].toarray().ravel()
                hit = at != 0
                assert np.array_equal(got[~hit], plain[~hit]), j
                assert np.array_equal(got[hit], np.sign(at[hit]) * value, equal_nan=True), j
    ws.close()
