"""CTA pairs on 256 x 192 tiles whose last tile of a row stores an odd number of chunks: the warps that alternate between two staging
buffers go on with the one that the last store does not read. (A product that ends up short of time shows it: many tiles, short K.)"""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,f32", [(4100, False), (1024, False), (4128, True), (4000, True)])
@pytest.mark.parametrize("gs_mode", [0, 1])
def test_no_chunk_overwrites_one_that_is_being_stored(N, f32, gs_mode):
    from paper_2510_27527_b200 import binding as b

    g = torch.Generator(device="cuda").manual_seed(N)
    A, W = (b.nvfp4_quantize(torch.randn(r, 128, device="cuda", generator=g).to(torch.bfloat16), gs_mode=gs_mode) for r in (9000, N))
    dt = b.DT_F32 if f32 else b.DT_BF16
    want = b.nvfp4_gemm_ex(A, W, dt, variant=b.GEMM_TILE128)
    for _ in range(30):
        assert torch.equal(b.nvfp4_gemm_ex(A, W, dt, variant=b.GEMM_PAIR192), want)
