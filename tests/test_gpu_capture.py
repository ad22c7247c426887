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


TWICE = SETUP + """
import ctypes
rt = ctypes.CDLL("libcudart.so.%s" % torch.version.cuda.split(".")[0])
def ok(rc):
    assert rc == 0, rc
s = torch.cuda.Stream()
st = ctypes.c_void_p(s.cuda_stream)
graph, execs = ctypes.c_void_p(), [ctypes.c_void_p(), ctypes.c_void_p()]
ok(rt.cudaStreamBeginCapture(st, 0))
msg.sample_field(prep, npts, M, mode, xi, Z, stream=s)
ok(rt.cudaStreamEndCapture(st, ctypes.byref(graph)))
for e in execs:
    ok(rt.cudaGraphInstantiate(ctypes.byref(e), graph, ctypes.c_ulonglong(0)))
for e in execs:
    Z.zero_()
    torch.cuda.synchronize()
    ok(rt.cudaGraphLaunch(e, st))
    s.synchronize()
    got = Z.clone()
msg.sample_field(prep, npts, M, mode, xi, Z)
torch.cuda.synchronize()
assert torch.equal(got, Z)
"""


def test_captured_fp32_call_allocates_nothing():
    """Its graph can be instantiated twice, which one with an allocation cannot."""
    _run(TWICE, "FP32")
