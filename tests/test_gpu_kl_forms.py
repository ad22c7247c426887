"""Every form of the FP32 contraction (three sample tiles, coefficients formed in the tile
or before it) at sizes with ragged tiles: within the FP32 bound of FP64, (M + 4) 2^-24 of
sum_m |Phi sqrt(lambda) xi|, and with the bits that the first samples have in a small call."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"

# narrow tiles direct and not, middle tiles direct and not, wide tiles direct and not
SIZES = [(401, 64, 333), (401, 401, 333), (11525, 70, 101), (11525, 250, 50), (40001, 3, 500), (40001, 37, 500)]


@pytest.mark.parametrize("npts,M,S", SIZES)
def test_forms_agree(npts, M, S):
    from paper_1907_12334_gb300 import build, msg

    build.build()
    g = torch.Generator(device=DEV).manual_seed(npts + M + S)
    Phi = torch.randn(npts, M, dtype=torch.float64, device=DEV, generator=g)
    sl = torch.rand(M, dtype=torch.float64, device=DEV, generator=g) + 0.1
    xi = torch.randn(S, M, dtype=torch.float64, device=DEV, generator=g)
    prep = torch.empty(msg.kl_prepared_bytes(npts, M, msg.MSG_GEMM_FP32), dtype=torch.uint8, device=DEV)
    msg.kl_prepare(Phi, sl, msg.MSG_GEMM_FP32, prep)

    def field(n):
        Z = torch.full((n, npts), float("nan"), dtype=torch.float64, device=DEV)
        msg.sample_field(prep, npts, M, msg.MSG_GEMM_FP32, xi[:n].contiguous(), Z)
        return Z

    Z = field(S)
    assert torch.equal(Z[:5], field(5))
    ref, scale = (xi * sl) @ Phi.T, (xi * sl).abs() @ Phi.abs().T
    assert bool(((Z - ref).abs() <= (M + 4) * 2.0 ** -24 * scale).all())


@pytest.mark.parametrize("mode", ["FP32", "FP64"])
def test_rows_of_many_terms(mode):
    """A tile of points whose rows hold more than 2^31 terms together (its last row starts
    beyond a 32-bit offset).  Few nonzero coefficients and a basis of small whole numbers: exact."""
    from paper_1907_12334_gb300 import build, msg

    build.build()
    npts, M, m = 128, 17_000_003, getattr(msg, f"MSG_GEMM_{mode}")
    Phi = torch.arange(npts, dtype=torch.float64, device=DEV)[:, None] + torch.arange(M, dtype=torch.float64, device=DEV)[None]
    Phi.remainder_(7)
    at = torch.tensor([0, 15, 16, 12_345_678, M - 17, M - 2, M - 1], device=DEV)
    xi = torch.zeros(1, M, dtype=torch.float64, device=DEV)
    xi[0, at] = torch.arange(1, 8, dtype=torch.float64, device=DEV)
    sl = torch.ones(M, dtype=torch.float64, device=DEV)
    prep = torch.empty(msg.kl_prepared_bytes(npts, M, m), dtype=torch.uint8, device=DEV)
    msg.kl_prepare(Phi, sl, m, prep)
    Z = torch.empty(1, npts, dtype=torch.float64, device=DEV)
    msg.sample_field(prep, npts, M, m, xi, Z)
    assert torch.equal(Z[0], Phi[:, at] @ xi[0, at])
