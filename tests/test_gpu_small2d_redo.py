"""FP64 wave solves of small order-2 2D grids whose waits run out: the limit reaches
them, the give-ups are counted, and applies, right-hand sides and solves keep
their results to the bit (one CTA redoes the solve without waits)."""
import numpy as np
import pytest

from paper_2205_12344_gb300 import inputs
from _helpers import to_np

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


@pytest.mark.parametrize("nu,bc,nrhs", [([2, 2], [D] * 4, 1), ([40, 34], [D, D, D, F], 1), ([33, 47], [F] * 4, 3),
                                        ([131, 94], [F, D, F, D], 1)])
def test_fp64_solve_survives_waits_that_run_out(nu, bc, nrhs):
    from paper_2205_12344_gb300 import _lib as L
    from paper_2205_12344_gb300.api import WaveHoltz
    p = inputs.small_problem(2, nu, 2, bc + [0, 0], seed=42, nrhs=nrhs)
    v = inputs.random_vectors(p, 1, 61)[0]
    ctas = nu[0] * nu[1] > 4  # one CTA per right-hand side waits for nobody
    with WaveHoltz(p) as wh:
        good, pi0 = to_np(wh.apply_S(v)), to_np(wh.apply_Pi0())
        x, info = wh.solve(tol=1e-9, raise_on_error=False)
        x = to_np(x)
        assert L.ewh_get_info(wh.ctx).kernel_variant[0] == 3 and np.isfinite(good).all()
        wh.reset_stats()
        wh.set_grid_wait(0)
        assert np.array_equal(to_np(wh.apply_S(v)), good) and np.array_equal(to_np(wh.apply_Pi0()), pi0)
        if ctas:
            assert wh.stats().grid_wait_timeouts == 2
        again, info2 = wh.solve(tol=1e-9, raise_on_error=False)
        assert np.array_equal(to_np(again), x) and info2.iters == info.iters and info2.status == info.status
        wh.set_grid_wait(10 ** 9)
        n = wh.stats().grid_wait_timeouts
        assert np.array_equal(to_np(wh.apply_S(v)), good) and wh.stats().grid_wait_timeouts == n
