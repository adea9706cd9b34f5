"""The launches that run several quantizers of a layer call at once, against the entry points that run them one by one: the same
bytes in every operand (padding of the scales included), scale and output."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def B():
    from paper_2510_27527_b200 import binding

    return binding


def poison(ws):
    ws.fill_(0xA5)
    return ws


# one row; less than a tile; one more than a tile in every direction; k blocks that end inside a 256-wide k tile; whole tiles; the
# last sizes within the limit of the fused backward and the first ones past it on 148 SMs (TENSOR: 19 CTAs per SM, 2812; BLOCK128: 5,
# 740): 3300 and 3500 x 1024 x 3072 have 2667 and 2833 CTAs (Q3 a CTA per 256 units of 64, the others per 128 x 64 tile), 1900 and
# 2000 x 1024 x 1024 have 727 and 765
SHAPES = [(1, 8, 8), (5, 40, 24), (127, 72, 136), (129, 136, 264), (257, 520, 392), (256, 512, 512), (384, 1032, 1288), (3000, 1024, 3072),
          (1024, 1024, 3080), (3300, 1024, 3072), (3500, 1024, 3072), (1900, 1024, 1024), (2000, 1024, 1024)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("gs_mode,rht", [(0, False), (0, True), (1, False), (2, False), (2, True)])
def test_layer_equals_separate_calls(shape, gs_mode, rht):
    b = B()
    T, D, C = shape
    g = torch.Generator(device="cuda").manual_seed(T + D + C)
    mk = lambda r, c, s: (torch.randn(r, c, generator=g, device="cuda") * s).bfloat16()
    x, w, dy = mk(T, D, 1.0), mk(C, D, 0.02), mk(T, C, 1e-4)
    x[-1, -1] = 9.0  # the maximum in the last element
    dy[-1, -1] = -3.0
    cfg = b.LayerConfig(gs_mode=gs_mode, seed=11, rht=rht)
    cfg.prepare(D)
    saved = b.alloc_saved(x, w, cfg)
    for q in (saved.qx, saved.qw):
        q.codes.fill_(0xA5), q.sf.fill_(0xA5)
    y, _ = b.nvfp4_linear_fwd(x, w, cfg, saved=saved, workspace=poison(b.linear_workspace(b.OP_FWD, T, D, C, cfg)))
    for q, src, sid in ((saved.qx, x, 1), (saved.qw, w, 2)):
        one = b.nvfp4_quantize(src, seed=11, stream_id=sid, gs_mode=gs_mode, out=b.alloc_operand(q.R, q.K, gs_mode, poison=True))
        assert torch.equal(q.codes, one.codes) and torch.equal(q.sf, one.sf) and torch.equal(q.gscale, one.gscale)
    ws = poison(b.linear_workspace(b.OP_BWD, T, D, C, cfg))
    dx, dw = b.nvfp4_linear_bwd(dy, saved, cfg, workspace=ws)
    wx, ww = poison(b.linear_workspace(b.OP_BWD_DX, T, D, C, cfg)), poison(b.linear_workspace(b.OP_BWD_DW, T, D, C, cfg))
    dx1 = b.nvfp4_linear_bwd_dx(dy, saved, cfg, workspace=wx)
    dw1 = b.nvfp4_linear_bwd_dw(dy, saved, cfg, workspace=ww)
    torch.cuda.synchronize()
    for which in (3, 4, 5, 6):
        f = b.nvfp4_linear_bwd_operand(b.OP_BWD, which, T, D, C, cfg, ws)
        o = b.nvfp4_linear_bwd_operand(b.OP_BWD_DX if which <= 4 else b.OP_BWD_DW, which, T, D, C, cfg, wx if which <= 4 else ww)
        assert torch.equal(f.codes, o.codes), f"Q{which} codes"
        assert torch.equal(f.sf, o.sf), f"Q{which} scales"
        assert torch.equal(f.gscale, o.gscale), f"Q{which} global scales"
    assert torch.equal(dx, dx1) and torch.equal(dw, dw1)


@pytest.mark.parametrize("rows,cols", [(1, 8), (64, 4096), (64, 4104), (65, 4096), (513, 4096), (2049, 4104), (4200, 4104)])
@pytest.mark.parametrize("where", [0, -1])
@pytest.mark.parametrize("pad", [0, 8])
def test_tensor_maximum(rows, cols, where, pad):
    """One CTA, as many CTAs as words, clusters of eight (part idle; 33; as many clusters as words): the scale is the maximum's."""
    b = B()
    buf = torch.zeros(rows, cols + pad, dtype=torch.bfloat16, device="cuda")
    x = buf[:, :cols]
    x.fill_(0.5)
    x[0 if where == 0 else rows - 1, 0 if where == 0 else cols - 1] = -21.0
    if pad:
        buf[:, cols:] = 1000.0  # not part of the matrix
    q = b.nvfp4_quantize(x, gs_mode=b.GS_TENSOR, workspace=poison(torch.empty(256, dtype=torch.uint8, device="cuda")))
    torch.cuda.synchronize()
    assert q.gscale.item() == (torch.tensor(21.0) / torch.tensor(2688.0)).item()


@pytest.mark.parametrize("rows", [513, 517, 1025, 4097])  # one row past whole clusters: most CTAs of the last one have nothing to read
def test_tensor_maximum_with_ctas_that_have_no_work(rows):
    b = B()
    xs = [torch.full((rows, 4096), 0.5, dtype=torch.bfloat16, device="cuda") for _ in range(4)]
    ends = torch.tensor([3.0, -21.0, 5.0, -40.0])
    for x, v, i in zip(xs, ends.tolist(), (0, rows - 1, rows // 2, rows - 1)):
        x[i, -1] = v
    ops = [[b.alloc_operand(rows, 4096, b.GS_TENSOR) for _ in xs] for _ in range(10)]
    ws = torch.empty(256, dtype=torch.uint8, device="cuda")
    for row in ops:  # back to back on one workspace
        for x, q in zip(xs, row):
            b.nvfp4_quantize(x, gs_mode=b.GS_TENSOR, out=q, workspace=ws)
    torch.cuda.synchronize()
    want = (ends.abs() / torch.tensor(2688.0)).tolist()
    for row in ops:
        assert [q.gscale.item() for q in row] == want
