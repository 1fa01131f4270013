"""The 2D order-2 level (tiles of 32 columns): tile remainders, every side type,
several right-hand sides, both precisions, the operator alone."""
import numpy as np
import pytest

from oracle import ewh_oracle as O
from paper_2205_12344_gb300 import inputs
from _helpers import oracle_all_rhs, rel_err, to_np, tol32

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

D, F = inputs.DIRICHLET, inputs.FREE


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_12344_gb300 import build
    build.build()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("nu,bc,nrhs", [([2, 2], [D] * 4, 1), ([31, 9], [F] * 4, 2), ([33, 8], [D, D, D, F], 1),
                                        ([64, 17], [F, D, D, F], 3), ([30, 62], [D, F, F, D], 1)])
def test_order2_2d_matches_oracle(nu, bc, nrhs, precision, monkeypatch):
    from paper_2205_12344_gb300.api import WaveHoltz
    monkeypatch.setenv("EWH_AUTOTUNE", "0")  # tiles of 8 rows
    p = inputs.small_problem(2, nu, 2, bc + [0, 0], seed=nu[0], nrhs=nrhs)
    s = O.build_system(p)
    v = inputs.random_vectors(p, 1, 3)[0]
    tol = 1e-12 if precision == "fp64" else tol32(s.nt)
    with WaveHoltz(p, precision=precision) as wh:
        got, pi0 = to_np(wh.apply_S(v)), to_np(wh.apply_Pi0())
        k = to_np(wh.apply_minvK(v))
    assert rel_err(got, oracle_all_rhs(s, lambda ss, x, r: O.apply_S(ss, x, r), v)) < tol
    assert rel_err(pi0, np.concatenate([O.apply_Pi0(s, r) for r in range(nrhs)])) < tol
    assert rel_err(k, oracle_all_rhs(s, lambda ss, x, r: O.minv_K(ss, x), v)) < 1e-12
