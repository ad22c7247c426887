"""The on-chip cycles (csrc/mid.cuh) against the phase-by-phase kernels.

``tune_low_cut`` = 4 keeps the recursion below diagonal 4 as table phases and
every stage on the host schedule; the default runs stages up to 9 (FP64: 8) whole
in one kernel, the recursion below diagonal 6 of larger items in another, and the
calls on diagonal 3 as one matrix.  Both iterate every grid to the same residual,
so Q agrees to what that residual allows (1e-8 relative, the mixed path's
tolerance; FP64 cycles 1e-10), and the cycle counts to one cycle wherever eps lies
above the rounding floor of the FP64 residual (below it, rounding decides the stop):
the floor is 2^-52 |A| |u| with |A| <= 2 a_max (4^p + 4^q) and |u| <= 1 / (8 a_min).
"""
import numpy as np
import pytest

import oracle
from paper_1907_12334_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"

# one-column and one-row hierarchies, each clipped triangle of the matrix, the
# last stage of k_item and the first ones after it, wide and tall
SHAPES = [(1, 1), (1, 5), (5, 1), (2, 4), (4, 2), (3, 3), (4, 5), (5, 6), (1, 10), (10, 1), (6, 6), (7, 5), (2, 9)]


@pytest.mark.parametrize("mu,nu1,nu2,precision", [(2, 2, 2, "MIXED"), (1, 1, 1, "MIXED"), (3, 2, 1, "MIXED"),
                                                  (2, 0, 3, "MIXED"), (2, 3, 0, "MIXED"), (2, 2, 2, "FP64"),
                                                  (1, 0, 2, "FP64")])
def test_on_chip_cycles_match_the_phase_kernels(mu, nu1, nu2, precision):
    from paper_1907_12334_gb300 import build, msg

    build.build()
    Z = torch.from_numpy(np.concatenate([inputs.smooth_field(P, Q, 1.5) for P, Q in SHAPES])).to(DEV)
    pq = np.array(SHAPES, dtype=np.int32)
    kw = dict(mu=mu, nu1=nu1, nu2=nu2, eps=1e-11, max_cycles=400, precision=getattr(msg, f"MSG_PREC_{precision}"))
    a = [t.cpu().numpy() for t in msg.solve(pq, Z, msg.SolverParams(**kw))]
    b = [t.cpu().numpy() for t in msg.solve(pq, Z, msg.SolverParams(tune_low_cut=4, **kw))]
    assert np.array_equal(a[1], b[1])
    np.testing.assert_allclose(a[0], b[0], rtol=1e-8 if precision == "MIXED" else 1e-10)
    k = 0
    for P, Q in SHAPES:
        contrast = np.exp(np.ptp(inputs.smooth_field(P, Q, 1.5)))
        for p in range(1, P + 1):
            for q in range(1, Q + 1):
                floor = 2.0 ** -52 * 2 * contrast * (4.0 ** p + 4.0 ** q) / 8
                assert floor > kw["eps"] or abs(int(a[2][k]) - int(b[2][k])) <= 1, (P, Q, p, q)
                k += 1


@pytest.mark.parametrize("P,Q,kw", [(5, 6, {}), (7, 4, dict(nu1=1, nu2=3)), (9, 2, {}), (2, 9, dict(mu=1)), (6, 6, dict(nu1=0)),
                                    (1, 10, {})])
def test_history_beyond_one_cta_matches_oracle(P, Q, kw):
    """Residual histories on hierarchies that run on launches of visits and k_mid: both
    sides in FP64, so they agree to 1e-8 relative down to the residual's rounding floor
    (as above, four times: two sides, and rounding of u beside that of the residual)."""
    from paper_1907_12334_gb300 import build, msg

    build.build()
    n, Z = 6, inputs.smooth_field(P, Q, 1.0)
    h = msg.msg_cycle_history(P, Q, 2, msg.SolverParams(**kw), 0, torch.from_numpy(np.concatenate([Z, -Z])).to(DEV), n)
    floor = 2.0 ** -52 * 2 * np.exp(np.ptp(Z)) * (4.0 ** P + 4.0 ** Q) / 8
    prm = msg.SolverParams(**kw)
    op = oracle.SolverParams(mu=prm.mu, nu1=prm.nu1, nu2=prm.nu2, omega=prm.omega)
    for k, z in enumerate((Z, -Z)):
        ho = oracle.Hierarchy(P, Q, Z=z, prm=op).cycle_history(0, n)
        np.testing.assert_allclose(h[k].cpu().numpy(), ho, rtol=1e-8, atol=4 * floor)


@pytest.mark.parametrize("P,Q,S,precision", [(8, 8, 160, "MIXED"), (6, 9, 40, "MIXED"), (7, 6, 40, "FP64"), (5, 5, 8, "MIXED")])
def test_workspace_contents_do_not_matter(P, Q, S, precision):
    """A workspace full of NaN gives the bits that one full of zeros gives (nothing is read
    before it is written, also with weight zero)."""
    from paper_1907_12334_gb300 import build, msg

    build.build()
    pq = np.array([(P, Q)] * S, dtype=np.int32)
    z = torch.from_numpy(inputs.smooth_field(P, Q, 1.5)).to(DEV)
    Z = (z[None] * torch.linspace(-1, 1, S, dtype=torch.float64, device=DEV)[:, None]).reshape(-1).contiguous()
    prm = msg.SolverParams(eps=1e-9, max_cycles=60, precision=getattr(msg, f"MSG_PREC_{precision}"))
    n, _ = msg.packed_sizes(pq)
    out = []
    for fill in (0, 255, 255):
        ws = torch.full((msg.msg_workspace_bytes(pq, prm),), fill, dtype=torch.uint8, device=DEV)
        Q_, st = torch.empty(n, dtype=torch.float64, device=DEV), torch.empty(S, dtype=torch.int32, device=DEV)
        msg.msg_solve_batch(pq, prm, Z, Q_, st, workspace=ws)
        out.append((Q_.cpu(), st.cpu()))
    assert int(out[0][1].abs().max()) == 0
    for q, st in out[1:]:
        assert torch.equal(q, out[0][0]) and torch.equal(st, out[0][1])
