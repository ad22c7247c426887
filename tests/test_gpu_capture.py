"""sample_field under stream capture, as the first call of its process (nothing the library
makes on first use may end the capture): the replayed graph gives an uncaptured call's bits."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

pytest.importorskip("torch")

SETUP = """
import sys, torch
from paper_1907_12334_gb300 import msg
mode = getattr(msg, "MSG_GEMM_" + sys.argv[1])
npts, M, S = 20000, 100, 300
g = torch.Generator(device="cuda:0").manual_seed(1)
Phi, xi = (torch.randn(n, M, dtype=torch.float64, device="cuda:0", generator=g) for n in (npts, S))
prep = torch.empty(msg.kl_prepared_bytes(npts, M, mode), dtype=torch.uint8, device="cuda:0")
msg.kl_prepare(Phi, torch.ones(M, dtype=torch.float64, device="cuda:0"), mode, prep)
Z = torch.zeros(S, npts, dtype=torch.float64, device="cuda:0")
torch.cuda.synchronize()
"""
REPLAY = SETUP + """
G = torch.cuda.CUDAGraph()
with torch.cuda.graph(G):
    msg.sample_field(prep, npts, M, mode, xi, Z)
for _ in range(2):
    Z.fill_(float("nan"))
    G.replay()
torch.cuda.synchronize()
got = Z.clone()
msg.sample_field(prep, npts, M, mode, xi, Z)
msg.msg_device_status()
assert torch.equal(got, Z)
"""


def _run(script, mode):
    from paper_1907_12334_gb300 import build

    build.build()
    r = subprocess.run([sys.executable, "-c", script, mode], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]


@pytest.mark.parametrize("mode", ["FP32", "BF16X3", "TF32", "FP64"])
def test_first_call_can_be_captured(mode):
    _run(REPLAY, mode)
