"""msg_launch_count counts every kernel of a call, the ones in front of a contraction and the
start values of a convergence study included."""
import numpy as np
import pytest

from paper_1907_12334_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"


@pytest.mark.parametrize("mode,M,launches", [("FP32", 20, 1), ("FP32", 400, 2), ("FP64", 20, 1), ("BF16X3", 20, 2), ("TF32", 20, 2)])
def test_contraction(mode, M, launches):
    from paper_1907_12334_gb300 import build, msg

    build.build()
    m, npts = getattr(msg, f"MSG_GEMM_{mode}"), 400
    prep = torch.empty(msg.kl_prepared_bytes(npts, M, m), dtype=torch.uint8, device=DEV)
    one = torch.ones(npts, M, dtype=torch.float64, device=DEV)
    msg.kl_prepare(one, one[0].contiguous(), m, prep)
    n = msg.msg_launch_count()
    msg.sample_field(prep, npts, M, m, one[:8], torch.empty(8, npts, dtype=torch.float64, device=DEV))
    assert msg.msg_launch_count() - n == launches


def test_study_by_launches():
    from paper_1907_12334_gb300 import build, msg

    build.build()
    Z, n = torch.from_numpy(np.asarray(inputs.smooth_field(1, 10, 1.0))).to(DEV), [msg.msg_launch_count()]
    for cycles in (1, 2):
        msg.msg_cycle_history(1, 10, 1, msg.SolverParams(), msg.MSG_HIST_MSG, Z, cycles)
        n.append(msg.msg_launch_count())
    one, two = n[1] - n[0], n[2] - n[1]
    # before the cycles: coefficients, face image, matrices, start values, first norm
    assert one - (two - one) == 5
