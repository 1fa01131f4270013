"""The 3D FP32 z-march at the edges of its 64 x 8 and 32 x 8 tiles: last tiles
whose counts shift the tile origins, and z ranges that start or end inside the
closure planes of either side (EWH_ZM_GRID cuts the planes into shares)."""
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


@pytest.mark.parametrize("shape", ["zm16", "zm8"])
@pytest.mark.parametrize("nu,bc,cap", [([66, 10, 10], [D] * 6, 0), ([68, 12, 11], [D, D, D, D, F, F], 17),
                                       ([65, 9, 12], [F] * 6, 13), ([128, 8, 10], [D, F, F, D, F, D], 11),
                                       ([20, 11, 40], [D, D, D, D, F, F], 29)])
def test_tiles_and_shares_match_oracle(nu, bc, cap, shape, monkeypatch):
    from paper_2205_12344_gb300.api import WaveHoltz
    monkeypatch.setenv("EWH_STEP3D_O4", shape)
    if cap:
        monkeypatch.setenv("EWH_ZM_GRID", str(cap))
    p = inputs.small_problem(3, nu, 4, bc, seed=nu[0])
    s = O.build_system(p)
    v = inputs.random_vectors(p, 1, 3)[0]
    want = oracle_all_rhs(s, lambda ss, x, r: O.apply_S(ss, x, r), v)
    with WaveHoltz(p, precision="fp32") as wh:
        got, pi0 = to_np(wh.apply_S(v)), to_np(wh.apply_Pi0())
        assert np.array_equal(to_np(wh.apply_S(v)), got)
    assert rel_err(got, want) < tol32(s.nt)
    assert rel_err(pi0, O.apply_Pi0(s, 0)) < tol32(s.nt)
