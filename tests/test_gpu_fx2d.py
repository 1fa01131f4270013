"""The FP64 2D order-4 step in block fixed point: S applies against the oracle at
the edges of its tiles (32 x 16 and 32 x 8 nodes), every side type, media with
steep contrasts, several right-hand sides; values of any magnitude and
non-finite ones take the plain path."""
import numpy as np
import pytest

from oracle import ewh_oracle as O
from paper_2205_12344_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

D, F = inputs.DIRICHLET, inputs.FREE


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_12344_gb300 import build
    build.build()


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def _S(p, v):
    from paper_2205_12344_gb300.api import WaveHoltz
    with WaveHoltz(p) as wh:
        return wh.apply_S(v).cpu().numpy(), wh.apply_Pi0().cpu().numpy()


@pytest.mark.parametrize("shape", ["fx", "fx1"])
@pytest.mark.parametrize("nu,bc,nrhs", [((8, 8), (D, D, D, D), 1), ((34, 18), (D, D, D, D), 1), ((36, 20), (F, D, D, F), 2),
                                        ((33, 17), (F, F, F, F), 1), ((67, 35), (D, F, F, D), 1), ((31, 9), (D, F, D, F), 1),
                                        ((130, 50), (D, D, D, F), 3)])
def test_tiles_match_oracle(shape, nu, bc, nrhs, monkeypatch):
    monkeypatch.setenv("EWH_STEP2D_O4", shape)
    p = inputs.small_problem(2, list(nu), 4, list(bc), seed=nu[0] + nu[1], nrhs=nrhs)
    s = O.build_system(p)
    v = inputs.random_vectors(p, 1, 5)[0]
    n = p.n_unknowns()
    got, pi0 = _S(p, v)
    for r in range(nrhs):
        assert _rel(got[r * n:(r + 1) * n], O.apply_S(s, v[r * n:(r + 1) * n])) < 1e-12
        assert _rel(pi0[r * n:(r + 1) * n], O.apply_Pi0(s, r)) < 1e-12


@pytest.mark.parametrize("scale", [2.0 ** -500, 2.0 ** 500, 2.0 ** -960, 2.0 ** 1010])
def test_any_magnitude(scale, monkeypatch):
    """S is linear, and the steps take the field's scale out as a power of two: S (2^k v) = 2^k S v to FP64 rounding
    (2^-960: the scale in two factors; 2^1010: the plain path)."""
    monkeypatch.setenv("EWH_STEP2D_O4", "fx")
    p = inputs.small_problem(2, [40, 37], 4, [D, D, D, F], seed=2)
    v = inputs.random_vectors(p, 1, 6)[0]
    one, _ = _S(p, v)
    got, _ = _S(p, v * scale)
    assert _rel(got / scale, one) < 1e-12


@pytest.mark.parametrize("rows", [1, 19])
def test_contrast(rows, monkeypatch):
    """A few steep tiles take the plain path within a launch; a medium of them is left to the FP64 pair (1e-10: the
    stiff layer multiplies the number of levels)."""
    monkeypatch.setenv("EWH_STEP2D_O4", "fx")
    p = inputs.small_problem(2, [330, 37], 4, [D, D, D, F], seed=2)
    p.mu[:rows, :] *= 1e3
    s = O.build_system(p)
    v = inputs.random_vectors(p, 1, 6)[0]
    got, _ = _S(p, v)
    assert _rel(got, O.apply_S(s, v)) < 1e-10


@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_non_finite_values_spread_as_in_fp64(bad, monkeypatch):
    """At most as far as in the FP64 pair (whose closure rows also multiply their zero weights)."""
    p = inputs.small_problem(2, [70, 40], 4, [D, D, D, D], seed=3, omega=2e4)  # few levels reach far: NaN stays local
    from paper_2205_12344_gb300.api import WaveHoltz
    v = inputs.random_vectors(p, 1, 7)[0]
    v[5] = bad
    out = {}
    for shape in ("fx", "split"):
        monkeypatch.setenv("EWH_STEP2D_O4", shape)
        with WaveHoltz(p, nt=5) as wh:
            out[shape] = wh.apply_S(v).cpu().numpy()
    fin = {k: np.isfinite(o) for k, o in out.items()}
    assert not fin["fx"][5] and fin["split"].any() and fin["fx"][fin["split"]].all()
    assert np.allclose(out["fx"][fin["split"]], out["split"][fin["split"]], rtol=1e-11, atol=1e-12)


def test_zero_field_stays_zero(monkeypatch):
    monkeypatch.setenv("EWH_STEP2D_O4", "fx")
    p = inputs.small_problem(2, [40, 37], 4, [F, D, D, F], seed=4)
    got, _ = _S(p, np.zeros(p.n_unknowns()))
    assert not got.any()
