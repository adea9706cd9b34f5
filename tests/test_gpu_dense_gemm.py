"""The dense products of the simulated FP6 x FP4 layer on CTA pairs (256 x 256 and 256 x 192 tiles) and on 128 x 128 tiles: ragged edges
of the tiles in both directions, one k tile and many, several tiles per pair, guard columns."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [(2049, 2040, 64), (2300, 2056, 200), (3072, 1024, 640), (2817, 1000, 130), (4095, 3000, 256), (130, 257, 64),
                                   (3000, 1030, 700), (5000, 4100, 100)])
@pytest.mark.parametrize("f32", [True, False])
def test_dense_product_against_fp64(M, N, K, f32):
    from paper_2510_27527_b200 import binding as b

    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    mk = lambda r: (torch.randn(r, (K + 7) // 8 * 8, device="cuda", generator=g)).to(torch.bfloat16)[:, :K]  # noqa: E731
    A, W = b.nvfp4_fp6_quantize(mk(M)), b.nvfp4_fp6_quantize(mk(N))
    ld = (N + 7) // 8 * 8 + 8
    buf = torch.full((M, ld), 77.0, dtype=torch.float32 if f32 else torch.bfloat16, device="cuda")
    b.nvfp4_dense_gemm(A, W, b.DT_F32 if f32 else b.DT_BF16, out=buf[:, :N])
    a, w = A.vals.double() * A.gscale.double(), W.vals.double() * W.gscale.double()
    want, absdot = a @ w.T, a.abs() @ w.abs().T
    # exact products summed in FP32 (at most K roundings of 2^-24 of the sum of magnitudes) and scaled twice; then one rounding to BF16
    tol = (K + 3) * 2.0 ** -24 * absdot + (0.0 if f32 else 2.0 ** -8 * want.abs())
    assert bool(((buf[:, :N].double() - want).abs() <= tol).all())
    assert bool((buf[:, N:] == 77.0).all())
