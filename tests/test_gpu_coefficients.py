"""Coefficients from the shared table of exponentials (large batches) against those that
each grid forms itself (small batches): the same exponentials summed in the same order, so
Q, cycle counts and residuals agree bit for bit."""
import numpy as np
import pytest

from paper_1907_12334_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"

# one level along a direction, the smallest rectangle, slices that divide a grid or do not
SHAPES = [(1, 1), (1, 8), (8, 1), (2, 2), (2, 7), (6, 6), (5, 6), (6, 6), (7, 4), (6, 6), (3, 9), (6, 6)]


@pytest.mark.parametrize("coef", [0, 1])
@pytest.mark.parametrize("precision", ["MIXED", "FP64"])
def test_batch_has_the_bits_of_its_samples(coef, precision):
    from paper_1907_12334_gb300 import build, msg

    build.build()
    prm = msg.SolverParams(eps=1e-6, max_cycles=100, coef=coef, precision=getattr(msg, f"MSG_PREC_{precision}"))
    fields = [(-1) ** k * inputs.smooth_field(P, Q, 1.0 + 0.1 * k) for k, (P, Q) in enumerate(SHAPES)]
    a = msg.solve(np.array(SHAPES, dtype=np.int32), torch.from_numpy(np.concatenate(fields)).to(DEV), prm)
    b = [msg.solve(np.array([s], dtype=np.int32), torch.from_numpy(f).to(DEV), prm) for s, f in zip(SHAPES, fields)]
    for x, y in zip(a, zip(*b)):
        assert torch.equal(x, torch.cat(y))


def test_history_batch_has_the_bits_of_its_samples():
    from paper_1907_12334_gb300 import build, msg

    build.build()
    for method in (msg.MSG_HIST_MSG, msg.MSG_HIST_STANDARD):
        Z = [inputs.smooth_field(6, 5, 0.3 * k) for k in range(10)]
        a = msg.msg_cycle_history(6, 5, 10, msg.SolverParams(), method, torch.from_numpy(np.concatenate(Z)).to(DEV), 4)
        for k, z in enumerate(Z):
            b = msg.msg_cycle_history(6, 5, 1, msg.SolverParams(), method, torch.from_numpy(z).to(DEV), 4)
            assert torch.equal(a[k], b[0])
