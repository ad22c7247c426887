"""Launch shapes where they are read, and the visits against kernels that share none of their code.

Stages up to 9 (FP64: 8) run whole on chip and read no launch shape, so the shapes of the
phase kernel are compared with ``tune_low_cut`` set, and ``tune_block`` on hierarchies with
visits: grids of one CTA, of clusters, of slabs down to two rows, thin grids that a cluster
cannot slice, and (FP64) grids beyond the largest cluster.  Launch shapes regroup
independent updates, so the results are equal bit for bit.

The other arm of the comparison of visits (``tune_low_cut`` = 4, ``tune_visit_smem`` = 2) runs the
table phases and the register-cached and global-memory visits instead of k_mid and k_visit.
Both iterate each grid to a relative residual of eps, so u differs by at most 2 eps / (16 a_min)
and Q, at least 1 / (64 a_max), by 8 eps contrast relatively; cycle counts differ by at most
one wherever eps lies above the rounding floor of the FP64 residual, 2^-52 |A| |u| with
|A| <= 2 a_max (4^p + 4^q) and |u| <= 1 / (8 a_min).
"""
import numpy as np
import pytest

import oracle
from paper_1907_12334_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"


def _solve(shapes, amp, **kw):
    from paper_1907_12334_gb300 import build, msg

    build.build()
    if "precision" in kw:
        kw["precision"] = getattr(msg, "MSG_PREC_" + kw["precision"])
    Z = np.concatenate([(-1) ** k * inputs.smooth_field(P, Q, amp) for k, (P, Q) in enumerate(shapes)])
    r = msg.solve(np.array(shapes, dtype=np.int32), torch.from_numpy(Z).to(DEV), msg.SolverParams(**kw))
    return [t.cpu().numpy() for t in r]


def _equal(a, b):
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("shape", [dict(tune_low_warps=3), dict(tune_low_items=1), dict(tune_low_items=4, tune_low_warps=1),
                                   dict(tune_low_items=8, tune_low_warps=1), dict(tune_block=64, tune_low_warps=1)])
def test_phase_kernel_shapes_do_not_change_results(shape):
    shapes = [(1, 1), (1, 4), (4, 1), (2, 3), (3, 5), (5, 5), (4, 4), (2, 6), (6, 2), (5, 4), (7, 4)]
    kw = dict(eps=1e-10, max_cycles=300, tune_low_cut=4)
    _equal(_solve(shapes, 1.0, **kw), _solve(shapes, 1.0, **kw, **shape))


@pytest.mark.parametrize("precision,shapes", [("MIXED", [(7, 6), (8, 8), (11, 2), (12, 2), (7, 6)]), ("FP64", [(6, 6), (11, 2), (7, 8)])])
def test_visit_block_does_not_change_results(precision, shapes):
    kw = dict(eps=1e-8, max_cycles=100, precision=precision)
    ref = _solve(shapes, 0.5, **kw)
    for block in (32, 64, 256, 1024):
        _equal(ref, _solve(shapes, 0.5, tune_block=block, **kw))


@pytest.mark.parametrize("precision,shapes,amp,eps", [("MIXED", [(7, 6), (6, 8), (9, 5), (8, 8)], 1.5, 1e-10),
                                                      ("MIXED", [(11, 2), (12, 2), (2, 12)], 0.5, 1e-8),
                                                      ("FP64", [(6, 6), (5, 8), (7, 7), (8, 7)], 1.5, 1e-10),
                                                      ("FP64", [(11, 2), (2, 11)], 0.5, 1e-8)])
def test_visits_match_kernels_that_share_no_code(precision, shapes, amp, eps):
    kw = dict(eps=eps, max_cycles=100, precision=precision)
    a = _solve(shapes, amp, **kw)
    b = _solve(shapes, amp, tune_low_cut=4, tune_visit_smem=2, **kw)
    assert not a[1].any() and not b[1].any()
    o = 0
    for P, Q in shapes:
        contrast = np.exp(np.ptp(inputs.smooth_field(P, Q, amp)))
        at = slice(o, o + P * Q)
        np.testing.assert_allclose(a[0][at], b[0][at], rtol=8 * eps * contrast)
        p, q = np.arange(1, P + 1)[:, None], np.arange(1, Q + 1)[None]
        above = (2.0 ** -52 * 2 * contrast * (4.0 ** p + 4.0 ** q) / 8 < eps).ravel()
        assert (np.abs(a[2][at] - b[2][at])[above] <= 1).all(), (P, Q)
        o += P * Q


@pytest.mark.parametrize("P,Q,precision", [(12, 2, "MIXED"), (11, 2, "FP64")])
def test_diagonals_split_between_two_kernels_match_oracle(P, Q, precision):
    eps, contrast = 1e-8, np.exp(np.ptp(inputs.smooth_field(P, Q, 0.5)))
    a = _solve([(P, Q)], 0.5, eps=eps, max_cycles=100, precision=precision)
    res = oracle.solve_batch([(P, Q)], [inputs.smooth_field(P, Q, 0.5)], oracle.SolverParams(eps=eps, max_cycles=100))
    assert not a[1].any()
    np.testing.assert_allclose(a[0], res[0][0].ravel(), rtol=8 * eps * contrast)


@pytest.mark.parametrize("P,Q", [(10, 5), (8, 8)])
def test_history_on_the_largest_clusters_and_beyond_matches_oracle(P, Q):
    """FP64 grids in clusters of 16, and a top grid that no cluster takes: the tolerance of the
    histories beyond one CTA (relative 1e-8 down to four times the residual's rounding floor)."""
    from paper_1907_12334_gb300 import build, msg

    build.build()
    n, Z = 3, inputs.smooth_field(P, Q, 0.5)
    h = msg.msg_cycle_history(P, Q, 1, msg.SolverParams(), 0, torch.from_numpy(Z).to(DEV), n)
    ho = oracle.Hierarchy(P, Q, Z=Z, prm=oracle.SolverParams()).cycle_history(0, n)
    floor = 2.0 ** -52 * 2 * np.exp(np.ptp(Z)) * (4.0 ** P + 4.0 ** Q) / 8
    np.testing.assert_allclose(h[0].cpu().numpy(), ho, rtol=1e-8, atol=4 * floor)
