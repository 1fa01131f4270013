"""Non-finite activations and gradients in the convolutions spread as far as the definition
says and no further, also at the sides of images that no patch divides."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_12344_gb300 import build
    build.build()


def _wgrad(x, dy):
    """The definition: the sum over the pixels of the image, of the zero-padded x."""
    n, h, w, ci = x.shape
    out = np.zeros((dy.shape[3], 3, 3, ci))
    a = np.pad(x, ((0, 0), (1, 1), (1, 1), (0, 0)))
    with np.errstate(invalid="ignore"):
        for ky in range(3):
            for kx in range(3):
                out[:, ky, kx] = np.einsum("nhwo,nhwi->oi", dy, a[:, ky:ky + h, kx:kx + w])
    return out


@pytest.mark.parametrize("bad", [np.inf, np.nan])
@pytest.mark.parametrize("N,H,W,Ci,Co", [(2, 17, 9, 16, 16), (1, 19, 13, 64, 48), (1, 16, 8, 32, 32), (1, 31, 16, 96, 64)])
def test_weight_gradient(N, H, W, Ci, Co, bad):
    from paper_2205_12344_gb300 import _lib as L
    rng = np.random.default_rng(H + Co)
    xt = torch.tensor(rng.standard_normal((N, H, W, Ci)), dtype=torch.float32).to(torch.bfloat16)
    dyt = torch.tensor(rng.standard_normal((N, H, W, Co)), dtype=torch.float32).to(torch.bfloat16)
    xt[0, 3, W - 1, 2] = bad        # last column
    xt[N - 1, H - 1, 2, 5] = bad    # last row
    dyt[0, H - 1, W - 1, 7] = bad   # a corner of the gradient
    x, dy = (t.float().double().numpy() for t in (xt, dyt))
    xt, dyt = xt.cuda(), dyt.cuda()
    dw = torch.empty((Co, 3, 3, Ci), dtype=torch.float32, device="cuda")
    L.ewh_conv3x3_wgrad(xt, dyt, dw, N, H, W, Ci, Co)
    got, want = dw.cpu().double().numpy(), _wgrad(x, dy)
    assert np.array_equal(np.isfinite(got), np.isfinite(want))
    fin = np.isfinite(want)
    assert np.abs(got[fin] - want[fin]).max() < 1e-4 * np.abs(want[fin]).max()
    if bad == np.inf:
        inf = np.isinf(want)
        assert np.array_equal(got[inf], want[inf])
