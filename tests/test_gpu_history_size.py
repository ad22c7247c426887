"""A convergence study of more samples than a grid's second dimension holds, on a
hierarchy that runs by launches: every sample has the history it has in a study of three."""
import numpy as np
import pytest

from paper_1907_12334_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"


def test_study_of_66000_samples():
    from paper_1907_12334_gb300 import build, msg

    build.build()
    P, Q, S, n = 1, 10, 66000, 1
    Z = torch.from_numpy(np.stack([inputs.smooth_field(P, Q, a) for a in (0.5, 1.0, 1.5)])).to(DEV)
    few = msg.msg_cycle_history(P, Q, 3, msg.SolverParams(), msg.MSG_HIST_MSG, Z.reshape(-1), n)
    all_ = msg.msg_cycle_history(P, Q, S, msg.SolverParams(), msg.MSG_HIST_MSG, Z.repeat(S // 3, 1).reshape(-1), n)
    assert torch.equal(all_, few.repeat(S // 3, 1))
