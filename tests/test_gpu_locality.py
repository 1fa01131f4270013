"""A level of the explicit scheme is local: what lies outside a node's domain of
dependence (4 nodes a level at order 4) does not change a bit of it, however
large the values or stiff the medium there.  Arithmetic that scales a
neighbourhood by its largest value or modulus fails here."""
import numpy as np
import pytest

from paper_2205_12344_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

D, F = inputs.DIRICHLET, inputs.FREE
LEVELS = 5   # reach 20 nodes


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_12344_gb300 import build
    build.build()


@pytest.fixture(autouse=True, params=["tuned", "fx", "ym"])  # what EWH_STEP2D_O4 may name
def _one_kernel(request, monkeypatch, tmp_path):
    monkeypatch.setenv("EWH_TUNE_CACHE", str(tmp_path / "tune.json"))  # the second context takes the first one's choice
    if request.param != "tuned":
        monkeypatch.setenv("EWH_STEP2D_O4", request.param)


def _problem(mapped=False):
    p = inputs.small_problem(2, [300, 200], 4, [D, D, D, F], seed=3, omega=2e5)  # so few levels are stable
    if mapped:
        p.mapping = inputs.annulus_mapping(p.n, p.h)
    return p


def _S(p, v, precision):
    from paper_2205_12344_gb300.api import WaveHoltz
    with WaveHoltz(p, precision=precision, nt=LEVELS) as wh:
        return wh.apply_S(v).cpu().numpy().reshape(2, p.unknowns_per_axis()[1], p.unknowns_per_axis()[0])


@pytest.mark.parametrize("mapped", [False, True])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_small_values_next_to_a_large_one(precision, mapped):
    p = _problem(mapped)
    v = 1e-12 * inputs.random_vectors(p, 1, 7)[0]
    alone = _S(p, v, precision)
    w = v.copy()
    w[20 * p.unknowns_per_axis()[0]] = 1.0  # u at the first unknown of row 20
    both = _S(p, w, precision)
    assert np.array_equal(alone[:, :, 24:], both[:, :, 24:])
    assert not np.array_equal(alone[:, :, :4], both[:, :, :4])


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_soft_nodes_next_to_stiff_ones(precision):
    p = _problem()
    v = inputs.random_vectors(p, 1, 8)[0]
    soft = _S(p, v, precision)
    for a in (p.rho, p.lam, p.mu):
        a[:, :3] *= 40.0  # a strip of the same wave speed
    stiff = _S(p, v, precision)
    assert np.array_equal(soft[:, :, 24:], stiff[:, :, 24:])
