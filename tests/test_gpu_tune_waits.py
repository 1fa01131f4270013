"""A launch whose wait gives up ends early and leaves NaN: the autotuner must not
take its time for that of the kernel, nor keep it in the tuning file."""
import numpy as np
import pytest

from paper_2205_12344_gb300 import inputs
from _helpers import to_np

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

D, F = inputs.DIRICHLET, inputs.FREE


@pytest.mark.parametrize("dim,order,nu", [(2, 2, [62, 62]), (2, 4, [210, 190]), (3, 4, [70, 40, 30])])
def test_waits_that_run_out_while_tuning(dim, order, nu, monkeypatch, tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_12344_gb300 import _lib as L
    from paper_2205_12344_gb300 import build
    from paper_2205_12344_gb300.api import WaveHoltz
    build.build()
    monkeypatch.setenv("EWH_TUNE_CACHE", str(tmp_path / "tune.json"))
    p = inputs.small_problem(dim, nu, order, [D] * (2 * dim - 1) + [F], seed=4)
    v = inputs.random_vectors(p, 1, 5)[0]
    with WaveHoltz(p, precision="fp32") as wh:
        wh.set_grid_wait(0)
        assert np.isfinite(to_np(wh.apply_S(v))).all()
        chosen = L.ewh_get_info(wh.ctx).kernel_variant[1]
    assert chosen in ((0, 1, 2) if order == 2 else (0,))
    line = (tmp_path / "tune.json").read_text()
    assert line.rstrip("}\n ").endswith(": %d" % chosen)
