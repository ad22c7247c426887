"""The KL contraction at the edges of its tiles, every mode, against FP64.

Tolerances, per value of sum_m |Phi sqrt(lambda) xi|: an FP64 sum of M products in
any order (M + 2) 2^-53; FP32 products and sums in order, operands rounded once,
(M + 4) 2^-24; BF16X3 and TF32 as in test_gpu_parity.  An FP32 output adds its own
rounding.  Sizes: tiles of 128 points x 32, 64 or 128 samples and 16 terms (FP32), 32 x 8
and 64 terms (FP64), 256 x 128 and 64 or 32 terms (tensor cores, more tiles than SMs in
the last size), with rows of Phi that are and are not 16-byte aligned.
"""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"

SIZES = [(1, 1, 1), (127, 3, 31), (128, 16, 32), (129, 17, 33), (257, 64, 64), (300, 65, 65), (1000, 63, 128), (33, 401, 129),
         (11525, 70, 100), (90000, 36, 200)]


@pytest.mark.parametrize("npts,M,S", SIZES)
@pytest.mark.parametrize("mode", ["FP64", "FP32", "BF16X3", "TF32"])
@pytest.mark.parametrize("zf32,shift", [(False, 0), (True, 8)])
def test_contraction_at_tile_edges(npts, M, S, mode, zf32, shift):
    from paper_1907_12334_gb300 import build, msg

    build.build()
    m = getattr(msg, f"MSG_GEMM_{mode}")
    g = torch.Generator(device=DEV).manual_seed(npts + M + S)
    Phi = torch.randn(npts, M, dtype=torch.float64, device=DEV, generator=g)
    sl = torch.rand(M, dtype=torch.float64, device=DEV, generator=g) + 0.1
    xi = torch.randn(S, M, dtype=torch.float64, device=DEV, generator=g)
    if mode in ("BF16X3", "TF32"):
        shift = 0  # their prepared buffer is 256-byte aligned by contract (the others hold doubles: 8)
    n = msg.kl_prepared_bytes(npts, M, m)
    prep = torch.empty(n + shift, dtype=torch.uint8, device=DEV)[shift:]
    msg.kl_prepare(Phi, sl, m, prep)
    Z = torch.full((S, npts), float("nan"), dtype=torch.float32 if zf32 else torch.float64, device=DEV)
    msg.sample_field(prep, npts, M, m, xi, Z)
    msg.msg_device_status()
    ref, scale = (xi * sl) @ Phi.T, (xi * sl).abs() @ Phi.abs().T
    tol = {"FP64": (M + 4) * 2.0 ** -53, "FP32": (M + 4) * 2.0 ** -24, "BF16X3": 5e-5, "TF32": 1.2e-3}[mode]
    if zf32:
        tol += 2.0 ** -23
    assert bool(((Z.double() - ref).abs() <= tol * scale).all())
