"""Order-2 members of a batch, which keep the per-level tiles: they hold no workspace of
the on-chip solve, and a problem alone does not take over their tuning."""
import pytest

from paper_2205_12344_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

D = inputs.DIRICHLET


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_12344_gb300 import build
    build.build()


def _used(make):
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    held = make()
    torch.cuda.synchronize()
    used = free - torch.cuda.mem_get_info()[0]
    for h in held:
        h.close()
    return used


def test_members_hold_no_exchange_words():
    from paper_2205_12344_gb300.api import WaveHoltz, WaveHoltzBatch
    probs = [inputs.small_problem(2, [190, 190], 2, [D] * 4 + [0, 0], seed=k) for k in range(24)]
    _used(lambda: [WaveHoltz(probs[0])])  # the context's own memory
    alone = _used(lambda: [WaveHoltz(p) for p in probs])
    batch = _used(lambda: [WaveHoltzBatch(probs)])
    words = 190 * 190 * 2 * 2 * 2 * 8  # components, words a value, level parities
    assert alone - batch > len(probs) * words // 2


def test_tuning_of_members_is_kept_apart(monkeypatch, tmp_path):
    from paper_2205_12344_gb300 import _lib as L
    from paper_2205_12344_gb300.api import WaveHoltz, WaveHoltzBatch
    monkeypatch.setenv("EWH_TUNE_CACHE", str(tmp_path / "tune.json"))
    p = inputs.small_problem(2, [62, 62], 2, [D] * 4 + [0, 0], seed=1)
    v = inputs.random_vectors(p, 1, 2)[0]
    with WaveHoltzBatch([p]) as wb:
        b = wb.apply_S([v])[0].cpu()
        assert L.ewh_get_info(L.ewh_batch_member(wb.b, 0)).kernel_variant[0] in (0, 1, 2)
    with WaveHoltz(p) as wh:
        assert torch.equal(wh.apply_S(v).cpu(), b)  # every order-2 kernel gives the same bits
    keys = [k for k in (tmp_path / "tune.json").read_text().splitlines() if ":" in k]
    assert len(keys) == 2 and sum("|v6b|" in k for k in keys) == 1
