"""The 3D order-4 stress + divergence pair (nodes of a plane numbered row after
row): sizes at which a warp holds several rows or ends inside one, every side
type, both precisions, the operator alone."""
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
@pytest.mark.parametrize("nu,bc,nrhs", [([6, 6, 6], [D] * 6, 1), ([8, 9, 7], [F] * 6, 2), ([31, 33, 9], [D, F, F, D, D, F], 1),
                                        ([65, 7, 10], [D, D, D, D, F, D], 3)])
def test_pair_matches_oracle(nu, bc, nrhs, precision, monkeypatch):
    from paper_2205_12344_gb300.api import WaveHoltz
    monkeypatch.setenv("EWH_STEP3D_O4", "pair")
    p = inputs.small_problem(3, nu, 4, bc, seed=nu[0], nrhs=nrhs)
    s = O.build_system(p)
    v = inputs.random_vectors(p, 1, 3)[0]
    tol = 1e-12 if precision == "fp64" else tol32(s.nt)
    with WaveHoltz(p, precision=precision) as wh:
        got, pi0 = to_np(wh.apply_S(v)), to_np(wh.apply_Pi0())
        k = to_np(wh.apply_minvK(v))
    assert rel_err(got, oracle_all_rhs(s, lambda ss, x, r: O.apply_S(ss, x, r), v)) < tol
    assert rel_err(pi0, np.concatenate([O.apply_Pi0(s, r) for r in range(nrhs)])) < tol
    assert rel_err(k, oracle_all_rhs(s, lambda ss, x, r: O.minv_K(ss, x), v)) < 1e-12
