"""The on-chip wave solve of small order-2 2D grids (every level in one launch,
rims exchanged through tagged words): tiles from single warps to the largest,
remainders along both axes, every side type, several right-hand sides, both
precisions, repeated applies, and waits that run out."""
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


@pytest.fixture(autouse=True)
def _on_chip(monkeypatch):
    monkeypatch.setenv("EWH_STEP2D_O2", "r")


def variant(wh, precision):
    from paper_2205_12344_gb300 import _lib as L
    return L.ewh_get_info(wh.ctx).kernel_variant[0 if precision == "fp64" else 1]


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("nu,bc,nrhs", [([2, 2], [D] * 4, 1), ([3, 70], [F] * 4, 1), ([63, 61], [D] * 4, 1),
                                        ([64, 65], [F, D, D, F], 2), ([45, 47], [F, F, D, D], 5),
                                        ([131, 94], [D, D, D, F], 1), ([200, 203], [D, F, F, F], 1)])
def test_small2d_matches_oracle(nu, bc, nrhs, precision):
    from paper_2205_12344_gb300.api import WaveHoltz
    p = inputs.small_problem(2, nu, 2, bc + [0, 0], seed=nu[0], nrhs=nrhs)
    s = O.build_system(p)
    v = inputs.random_vectors(p, 1, 3)[0]
    tol = 1e-12 if precision == "fp64" else tol32(s.nt)
    with WaveHoltz(p, precision=precision) as wh:
        got, pi0 = to_np(wh.apply_S(v)), to_np(wh.apply_Pi0())
        assert variant(wh, precision) == 3
        again = to_np(wh.apply_S(v))
    assert rel_err(got, oracle_all_rhs(s, lambda ss, x, r: O.apply_S(ss, x, r), v)) < tol
    assert rel_err(pi0, np.concatenate([O.apply_Pi0(s, r) for r in range(nrhs)])) < tol
    assert np.array_equal(got, again)


def test_small2d_waits_that_run_out():
    from paper_2205_12344_gb300.api import WaveHoltz
    p = inputs.small_problem(2, [40, 34], 2, [D, D, D, F, 0, 0], seed=42)
    v = inputs.random_vectors(p, 1, 61)[0]
    with WaveHoltz(p, precision="fp32") as wh:
        good = to_np(wh.apply_S(v))
        assert variant(wh, "fp32") == 3
        wh.reset_stats()
        wh.set_grid_wait(0)
        assert np.isnan(to_np(wh.apply_S(v))).all()
        assert wh.stats().grid_wait_timeouts == 1
        x, info = wh.solve(tol=1e-8)  # finishes on the FP64 operator
        assert info.status == 0 and info.rel_res <= 1e-8
        wh.set_grid_wait(10 ** 9)
        assert np.array_equal(to_np(wh.apply_S(v)), good)
