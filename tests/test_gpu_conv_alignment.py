"""Operands of the convolutions off a 16-byte boundary: the weight gradient takes them
at any element, the others refuse them by name."""
import numpy as np
import pytest

from oracle import conv_oracle as C

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_12344_gb300 import build
    build.build()


def _bf(a, off):
    """FP64 array -> (BF16 view that starts `off` elements into its buffer, the same values in FP64)."""
    buf = torch.zeros(a.size + 8, dtype=torch.bfloat16, device="cuda")
    t = buf[off:off + a.size].view(a.shape)
    t.copy_(torch.tensor(a, dtype=torch.float32))
    assert t.data_ptr() % 16 == 2 * off
    return t, t.float().cpu().double().numpy()


@pytest.mark.parametrize("ox,od", [(1, 0), (0, 4), (3, 7)])
@pytest.mark.parametrize("N,H,W,Ci,Co", [(1, 1, 1, 16, 16), (2, 17, 9, 48, 80), (1, 40, 33, 64, 32)])
def test_weight_gradient_at_any_alignment(N, H, W, Ci, Co, ox, od):
    from paper_2205_12344_gb300 import _lib as L
    rng = np.random.default_rng(H + Co)
    xt, x = _bf(rng.standard_normal((N, H, W, Ci)), ox)
    dyt, dy = _bf(rng.standard_normal((N, H, W, Co)), od)
    dw = torch.full((Co, 3, 3, Ci), 3.0, dtype=torch.float32, device="cuda")  # overwritten
    L.ewh_conv3x3_wgrad(xt, dyt, dw, N, H, W, Ci, Co)
    ref = C.conv3x3_wgrad(x, dy)
    assert np.abs(dw.cpu().double().numpy() - ref).max() < 1e-4 * np.abs(ref).max()  # FP32 accumulation order


def test_unaligned_operands_are_refused_by_name():
    from paper_2205_12344_gb300 import _lib as L
    bad, _ = _bf(np.zeros((1, 8, 8, 16)), 1)
    wbad, _ = _bf(np.zeros((16, 3, 3, 16)), 4)
    x, w = torch.zeros_like(bad).contiguous(), torch.zeros_like(wbad).contiguous()
    out = torch.zeros((1, 8, 8, 16), dtype=torch.float32, device="cuda")
    for call in (lambda: L.ewh_conv3x3_fwd(bad, w, None, out, None, 0, 1, 8, 8, 16, 16),
                 lambda: L.ewh_conv3x3_fwd(x, wbad, None, out, None, 0, 1, 8, 8, 16, 16),
                 lambda: L.ewh_conv3x3_dgrad(bad, w, w.clone(), out, 1, 8, 8, 16, 16),
                 lambda: L.ewh_conv3x3_dgrad(x, w, wbad, out, 1, 8, 8, 16, 16)):
        with pytest.raises(RuntimeError, match="16-byte aligned"):
            call()
    torch.cuda.synchronize()
