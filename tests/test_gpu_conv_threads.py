"""The convolutions called from threads other than the one that set the GPU up: first calls of a
thread, one after another and of several threads at once (streams and buffers of their own)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = """
import sys, threading, torch
from paper_2205_12344_gb300 import _lib as L
L.load()
T = 16
x = [torch.ones((1, 16, 16, 16), dtype=torch.bfloat16, device="cuda") for _ in range(T)]
w = torch.ones((16, 3, 3, 16), dtype=torch.bfloat16, device="cuda")
out = [torch.zeros((1, 16, 16, 16), dtype=torch.float32, device="cuda") for _ in range(T)]
dw = [torch.zeros((16, 3, 3, 16), dtype=torch.float32, device="cuda") for _ in range(T)]
streams = [torch.cuda.Stream() for _ in range(T)]
torch.cuda.synchronize()
errors = []
def call(k, gate=None):
    if gate is not None: gate.wait()
    try:
        if sys.argv[1] != "wgrad":
            L.ewh_conv3x3_fwd(x[k], w, None, out[k], None, 0, 1, 16, 16, 16, 16, streams[k].cuda_stream)
        if sys.argv[1] != "fwd":
            L.ewh_conv3x3_wgrad(x[k], x[k], dw[k], 1, 16, 16, 16, 16, streams[k].cuda_stream)
    except Exception as e:
        errors.append(str(e))
if sys.argv[1] == "at once":
    sys.setswitchinterval(1e-6)
    gate = threading.Event()
    threads = [threading.Thread(target=call, args=(k, gate)) for k in range(T)]
    for t in threads: t.start()
    gate.set()
    for t in threads: t.join()
else:
    T = 1
    t = threading.Thread(target=call, args=(0,))
    t.start()
    t.join()
torch.cuda.synchronize()
assert not errors, errors
for k in range(T):
    assert sys.argv[1] == "wgrad" or float(out[k][0, 8, 8, 0]) == 144.0
    assert sys.argv[1] == "fwd" or float(dw[k][0, 1, 1, 0]) == 256.0
"""


def _run(how):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_12344_gb300 import build
    build.build()
    r = subprocess.run([sys.executable, "-c", PROGRAM, how], cwd=ROOT, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr[-2000:]


@pytest.mark.parametrize("how", ["fwd", "wgrad"])
def test_first_call_of_a_thread(how):
    _run(how)


@pytest.mark.parametrize("attempt", range(4))  # a race: one program shows it only now and then
def test_first_calls_of_several_threads(attempt):
    _run("at once")
