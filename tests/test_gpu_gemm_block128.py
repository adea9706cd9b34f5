"""The product with 1x128 outer scales at the sizes where its kernel can go wrong: edges of the 128 x 192, 128 and 64 tiles, tiles that
start in the middle of a 128-row scale tile, numbers of 128-k chunks around the groups of four (and rows of scales that cannot be read
in 16- or 8-byte pieces), several tiles per CTA."""
import pytest
import torch

pytestmark = pytest.mark.gpu
E2M1 = [0.0, 0.5, 1.0, 1.5, 2.0, 3.0, 4.0, 6.0]


def B():
    from paper_2510_27527_b200 import binding

    return binding


def dequantize(q):
    lut = torch.tensor(E2M1 + [-v for v in E2M1], dtype=torch.float64, device="cuda")
    c = q.codes.view(q.R, q.Kp // 2).long()
    v = torch.stack([lut[c & 15], lut[c >> 4]], -1).reshape(q.R, q.Kp)
    sf = torch.from_numpy(q.sf_linear()).cuda().view(torch.float8_e4m3fn).double()
    return v * sf.repeat_interleave(16, 1) * q.gscale.double().view(q.R, -1).repeat_interleave(128, 1)


@pytest.mark.parametrize("M,N,K", [(1, 8, 16), (128, 192, 128), (129, 193, 136), (127, 191, 256), (256, 384, 384), (130, 576, 512), (257, 448, 640),
                                   (64, 200, 896), (300, 328, 2816), (4100, 1160, 1000), (96, 64, 16384)])
@pytest.mark.parametrize("c_dtype", [0, 1])
@pytest.mark.parametrize("accumulate", [False, True])
def test_product(M, N, K, c_dtype, accumulate):
    b = B()
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    a = torch.randn(M, K, generator=g, device="cuda") * torch.exp2(torch.randint(-6, 7, (M, (K + 127) // 128), generator=g, device="cuda").float()
                                                                  ).repeat_interleave(128, 1)[:, :K]
    w = torch.randn(N, K, generator=g, device="cuda") * 0.02
    qa, qb = b.nvfp4_quantize(a.bfloat16(), gs_mode=b.GS_BLOCK128), b.nvfp4_quantize(w.bfloat16(), gs_mode=b.GS_BLOCK128)
    want = dequantize(qa) @ dequantize(qb).T
    ld = (N + 7) // 8 * 8 + 8
    buf = torch.full((M + 1, ld), 3.0, dtype=torch.float32 if c_dtype else torch.bfloat16, device="cuda")
    out = buf[:M, :N]
    if accumulate:
        old = (torch.randn(M, N, generator=g, device="cuda") * want.abs().mean()).to(buf.dtype)
        out.copy_(old)
        want = want + old.double()
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    b.nvfp4_gemm(qa, qb, c_dtype, out=out, accumulate=accumulate, dev_status=status)
    torch.cuda.synchronize()
    assert int(status) == 0
    assert bool((buf[M:] == 3.0).all()) and bool((buf[:, N:] == 3.0).all()), "outside C"
    # FP32: an element is a sum of G = K / 128 partials (exact products, at most 128 rounded additions each) with two roundings per
    # partial, so its error is below (128 + 2 + G) 2^-24 of the sum of magnitudes, which for random signs is about sqrt(K) of the
    # result: typical errors add in quadrature, sqrt(130 + G) 2^-24 sqrt(2) < 1.5e-6 of the norm. BF16 adds 2^-9.
    err = ((out.double() - want).norm() / want.norm()).item()
    assert err <= (3e-6 if c_dtype else 2.0**-9 + 3e-6), err


# the wide tiles, which products of few tiles do not take: 192 columns (whole and ragged last ones, starting in the middle of a scale
# tile; three chunks, five) and 128 (whole, ragged; eight chunks, three), in several rounds over the SMs
@pytest.mark.parametrize("M,N,K", [(2820, 1000, 392), (2700, 1152, 640), (2049, 1345, 136), (3000, 1160, 904), (9000, 1000, 304), (16400, 1024, 1000)])
@pytest.mark.parametrize("c_dtype", [0, 1])
@pytest.mark.parametrize("accumulate", [False, True])
def test_product_of_many_tiles(M, N, K, c_dtype, accumulate):
    test_product(M, N, K, c_dtype, accumulate)


@pytest.mark.parametrize("T,D,C", [(200, 264, 136), (2820, 384, 1000), (3000, 1000, 1160)])  # tiles of 64, 192 and 128 columns
def test_outlier_channels_ride_along(T, D, C):
    """The BF16 side product as one more partial: against the operands' product and X_out W_out^T in 64 bits."""
    b = B()
    g = torch.Generator(device="cuda").manual_seed(T)
    x, w = torch.randn(T, D, generator=g, device="cuda").bfloat16(), (torch.randn(C, D, generator=g, device="cuda") * 0.02).bfloat16()
    outl = list(range(3, D, 11))
    cfg = b.LayerConfig(gs_mode=b.GS_BLOCK128, outliers=outl, y_dtype=b.DT_F32)
    y, saved = b.nvfp4_linear_fwd(x, w, cfg)
    want = dequantize(saved.qx) @ dequantize(saved.qw).T + x[:, outl].double() @ w[:, outl].double().T
    assert ((y.double() - want).norm() / want.norm()).item() <= 3e-6  # (as above; the side product is one partial more)
