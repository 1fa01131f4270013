"""The tensor-core convolutions where their tiles can go wrong: images that no
8 x 16 patch divides, every channel block (16, 32, 64) and its multiples, output
channels that end inside a CTA's block, unaligned outputs; the clustered bias
gradient and the vectorised activation gradient at their limits.  Tolerances as
for the layer tests: the FP32 accumulation order is all that differs."""
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


def _bf(a):
    t = torch.tensor(a, dtype=torch.float32).to(torch.bfloat16).cuda().contiguous()
    return t, t.float().cpu().double().numpy()


def _rel(a, b):
    return np.abs(a - b).max() / max(np.abs(b).max(), 1e-30)


@pytest.mark.parametrize("N,H,W,Ci,Co,off", [(1, 1, 1, 16, 8, 0), (1, 16, 8, 64, 16, 0), (2, 17, 9, 48, 24, 1),
                                             (1, 5, 7, 96, 80, 0), (1, 33, 23, 192, 72, 1), (3, 15, 40, 128, 200, 0)])
def test_forward_tiles(N, H, W, Ci, Co, off):
    from paper_2205_12344_gb300 import _lib as L
    rng = np.random.default_rng(H * 100 + W)
    xt, x = _bf(rng.standard_normal((N, H, W, Ci)))
    wt, w = _bf(rng.standard_normal((Co, 3, 3, Ci)) / np.sqrt(9 * Ci))
    b = torch.tensor(rng.standard_normal(Co), dtype=torch.float32).cuda()
    pre = torch.full((N * H * W * Co + 2,), 7.0, dtype=torch.float32, device="cuda")
    act = torch.full((N * H * W * Co + 2,), 7.0, dtype=torch.bfloat16, device="cuda")
    n = N * H * W * Co
    L.ewh_conv3x3_fwd(xt, wt, b, pre[off:], act[off:], 1, N, H, W, Ci, Co)  # off = 1: not 16-byte aligned
    torch.cuda.synchronize()
    ref = C.conv3x3(x, w, b.cpu().double().numpy())
    assert _rel(pre[off:off + n].cpu().double().numpy().reshape(ref.shape), ref) < 2e-5
    assert _rel(act[off:off + n].float().cpu().double().numpy().reshape(ref.shape), C.leaky_relu(ref)) < 1e-2
    assert float(pre[off + n]) == 7.0 and float(act[off + n]) == 7.0  # nothing beyond the outputs


@pytest.mark.parametrize("N,H,W,Ci,Co", [(1, 1, 1, 16, 16), (1, 16, 8, 64, 64), (2, 17, 9, 48, 80), (1, 5, 7, 96, 32),
                                         (1, 33, 23, 192, 160), (3, 40, 70, 32, 16), (1, 18, 10, 16, 128)])
def test_gradient_tiles(N, H, W, Ci, Co):
    from paper_2205_12344_gb300 import _lib as L
    rng = np.random.default_rng(H * 100 + W + Co)
    xt, x = _bf(rng.standard_normal((N, H, W, Ci)))
    wt, w = _bf(rng.standard_normal((Co, 3, 3, Ci)) / np.sqrt(9 * Ci))
    dyt, dy = _bf(rng.standard_normal((N, H, W, Co)))
    dx = torch.empty((N, H, W, Ci), dtype=torch.float32, device="cuda")
    scratch = torch.empty(9 * Ci * Co, dtype=torch.bfloat16, device="cuda")
    L.ewh_conv3x3_dgrad(dyt, wt, scratch, dx, N, H, W, Ci, Co)
    dw = torch.full((Co, 3, 3, Ci), 3.0, dtype=torch.float32, device="cuda")  # overwritten
    L.ewh_conv3x3_wgrad(xt, dyt, dw, N, H, W, Ci, Co)
    torch.cuda.synchronize()
    assert _rel(dx.cpu().double().numpy(), C.conv3x3_dgrad(dy, w)) < 2e-5
    assert _rel(dw.cpu().double().numpy(), C.conv3x3_wgrad(x, dy)) < 1e-4


@pytest.mark.parametrize("P,Cc", [(1, 1), (127, 9), (16383, 20), (16384, 13), (50001, 32)])
def test_bias_gradient_clusters(P, Cc):
    from paper_2205_12344_gb300 import _lib as L
    g = torch.Generator(device="cuda").manual_seed(P)
    dy = torch.randn((P, Cc), dtype=torch.float32, device="cuda", generator=g) + 0.5
    out = []
    for _ in range(2):
        db = torch.empty(Cc, dtype=torch.float32, device="cuda")
        L.ewh_bias_grad(dy, db, P, Cc)
        out.append(db.cpu())
    assert torch.equal(out[0], out[1])  # a fixed order of additions
    ref = dy.double().sum(0).cpu().numpy()
    assert _rel(out[0].double().numpy(), ref) < 1e-5


@pytest.mark.parametrize("n,off", [(1, 0), (1027, 0), (1024, 1), (4099, 2)])
def test_activation_gradient_alignment(n, off):
    from paper_2205_12344_gb300 import _lib as L
    g = torch.Generator(device="cuda").manual_seed(n)
    pre, dy = (torch.randn(n + 4, dtype=torch.float32, device="cuda", generator=g)[off:off + n] for _ in range(2))
    dx = torch.zeros(n + 4, dtype=torch.float32, device="cuda")
    db = torch.zeros(n + 4, dtype=torch.bfloat16, device="cuda")
    L.ewh_leaky_relu_bwd(pre, dy, dx[off:], db[off:], n)
    torch.cuda.synchronize()
    want = torch.where(pre > 0, dy, dy * torch.tensor(0.1, dtype=torch.float32, device="cuda"))
    assert torch.equal(dx[off:off + n], want) and torch.equal(db[off:off + n], want.to(torch.bfloat16))
    assert float(dx[off + n:].abs().sum()) == 0.0 and float(db[off + n:].float().abs().sum()) == 0.0
