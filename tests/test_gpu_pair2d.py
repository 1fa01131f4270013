"""The stress + divergence pair of 2D order-4 grids (16-byte groups along x in the
rectangle of central differences, the frame node by node): every remainder of
a row against the group width, grids that are frame only, both low sides (the
rows' alignment), several right-hand sides, both precisions, the operator alone."""
import numpy as np
import pytest

from oracle import ewh_oracle as O
from paper_2205_12344_gb300 import inputs
from _helpers import TOL64, oracle_all_rhs, rel_err, to_np, tol32

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
@pytest.mark.parametrize("nu,bc,nrhs", [([6, 7], [D, D, D, D], 1), ([7, 9], [F, D, D, F], 2), ([8, 6], [D, F, F, D], 1),
                                        ([9, 20], [F, F, F, F], 1), ([10, 11], [D, F, D, F], 3), ([11, 31], [F, D, F, D], 1),
                                        ([70, 45], [D, D, D, F], 1), ([261, 157], [F, F, D, D], 2)])
def test_pair2d_matches_oracle(nu, bc, nrhs, precision, monkeypatch):
    from paper_2205_12344_gb300.api import WaveHoltz
    monkeypatch.setenv("EWH_STEP2D_O4", "split")
    p = inputs.small_problem(2, nu, 4, bc + [0, 0], seed=22, nrhs=nrhs)
    s = O.build_system(p)
    v = inputs.random_vectors(p, 1, 3)[0]
    with WaveHoltz(p, precision=precision) as wh:
        got, pi0, k = to_np(wh.apply_S(v)), to_np(wh.apply_Pi0()), to_np(wh.apply_minvK(v))
    tol = TOL64 if precision == "fp64" else tol32(s.nt)
    assert rel_err(got, oracle_all_rhs(s, lambda ss, x, r: O.apply_S(ss, x, r), v)) < tol
    assert rel_err(pi0, np.concatenate([O.apply_Pi0(s, r) for r in range(nrhs)])) < tol
    assert rel_err(k, oracle_all_rhs(s, lambda ss, x, r: O.minv_K(ss, x), v)) < 1e-12
