"""The implicit-GEMM convolutions (lbm_nn_conv3, lbm_nn_conv3_wgrad) at the edges of their tiles and
of their layouts (resident and staged weights, rolling and sequential planes, upsampled and joined
inputs, split outputs, the narrow first layer).

Both sum the same BF16 products in the same order as im2col rows and lbm_nn_gemm_tn, so they have to repeat
its results bit for bit."""
import numpy as np
import pytest

from oracle import nn_oracle as orc

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
from paper_2502_12955_gb300 import surrogate as sg  # noqa: E402


def _rand(shape, seed, dtype=torch.bfloat16):
    g = torch.Generator().manual_seed(seed)
    return torch.randn(shape, generator=g).to(dtype).cuda()


def _padded(x):
    x8 = torch.empty((x.shape[0], 8), dtype=torch.bfloat16, device="cuda")
    sg.lbm_nn_pad8(x, x8, x.shape[0], x.shape[1])
    return x8


# shapes (D, H, W): a partial tile along x and y, several z ranges per column, one plane, whole tiles
SHAPES = [(6, 16, 12), (16, 8, 8), (1, 16, 40), (40, 32, 16), (2, 20, 48)]
LAYERS = [(5, 0, 0, 16), (4, 0, 0, 48), (16, 0, 0, 16), (32, 0, 0, 32), (48, 0, 0, 64), (64, 0, 0, 224), (160, 0, 0, 160),
          (32, 1, 16, 16), (160, 1, 64, 64)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("ca,up,cb,co", LAYERS)
def test_conv3_repeats_the_im2col_gemm(shape, ca, up, cb, co):
    D, H, W = shape
    if up and (D | H | W) & 1:
        pytest.skip("upsampling needs even sizes")
    V, C = D * H * W, ca + cb
    assert V % 128 == 0 and sg.lbm_nn_conv3_fits(ca, up, cb, co)
    xa = _rand((V // 8 if up else V, ca), 1)
    xb = _rand((V, cb), 2) if cb else None
    w = _rand((co, C, 27), 3, torch.float32) * (2.0 / (27 * C)) ** 0.5
    bias = _rand((co,), 4, torch.float32)
    # rows
    x = xa
    if up:
        fine = torch.empty((V, ca), dtype=torch.bfloat16, device="cuda")
        sg.lbm_nn_up2(xa, fine, D // 2, H // 2, W // 2, ca, 0)
        x = torch.cat([fine, xb], 1).contiguous()
    kp = sg.kpad(27 * C)
    wk = torch.empty((co, kp), dtype=torch.bfloat16, device="cuda")
    sg.lbm_nn_pack_weights(w, wk, None, co, C, kp, 0)
    col = torch.empty((V, kp), dtype=torch.bfloat16, device="cuda")
    sg.lbm_nn_im2col(x, col, D, H, W, C, kp, 0)
    want = torch.empty((V, co), dtype=torch.bfloat16, device="cuda")
    sg.lbm_nn_gemm_tn(col, wk, want, co, V, co, kp, 1, sg.OUT_BF16_RELU, bias)
    if ca <= 8:
        xa = _padded(xa)
    # implicit, with the columns split over two outputs where there are several 16s
    wp = torch.empty(sg.lbm_nn_conv3_packed(co, C), dtype=torch.bfloat16, device="cuda")
    sg.lbm_nn_conv3_pack(w, wp, None, co, C)
    n0 = 16 if co > 16 else co
    y0 = torch.full((V, n0), float("nan"), dtype=torch.bfloat16, device="cuda")
    y1 = torch.full((V, co - n0), float("nan"), dtype=torch.bfloat16, device="cuda") if n0 < co else None
    sg.lbm_nn_conv3((xa, ca, up, xb, cb), shape, wp, co, y0, n0, y1, bias=bias, relu=1)
    sg.lbm_nn_status()
    got = torch.cat([y0, y1], 1) if y1 is not None else y0
    assert torch.equal(got, want)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("ca,up,cb,co", LAYERS)
def test_conv3_wgrad_repeats_the_split_gemm(shape, ca, up, cb, co):
    D, H, W = shape
    if up and (D | H | W) & 1:
        pytest.skip("upsampling needs even sizes")
    V, C = D * H * W, ca + cb
    xa = _rand((V // 8 if up else V, ca), 5)
    xb = _rand((V, cb), 6) if cb else None
    dy = _rand((V, co), 7)
    x = xa
    if up:
        fine = torch.empty((V, ca), dtype=torch.bfloat16, device="cuda")
        sg.lbm_nn_up2(xa, fine, D // 2, H // 2, W // 2, ca, 0)
        x = torch.cat([fine, xb], 1).contiguous()
    kp = sg.kpad(27 * C)
    col = torch.empty((kp, V), dtype=torch.bfloat16, device="cuda")
    sg.lbm_nn_im2col(x, col, D, H, W, C, kp, 1)
    splits = sg.lbm_nn_gemm_splits(V, max(1, min(64, (4 * 152) // ((kp // 128) * max(1, co // 128)), V // 64)))
    part = torch.empty((splits, kp, co), dtype=torch.float32, device="cuda")
    sg.lbm_nn_gemm_tn(col, dy.T.contiguous(), part, co, kp, co, V, splits, sg.OUT_F32, None)
    rows = torch.empty((kp, co), dtype=torch.float32, device="cuda")
    sg.lbm_nn_reduce_splits(part, rows, kp * co, splits, kp * co)
    want = torch.empty((co, C, 27), dtype=torch.float32, device="cuda")
    sg.lbm_nn_unpack_wgrad(rows, want, co, C)
    if ca <= 8:
        xa = _padded(xa)
    scratch = torch.empty(sg.lbm_nn_conv3_wgrad_scratch(shape, C, co), dtype=torch.float32, device="cuda")
    dw = torch.full((co, C, 27), float("nan"), dtype=torch.float32, device="cuda")
    sg.lbm_nn_conv3_wgrad((xa, ca, up, xb, cb), shape, dy, co, scratch, dw)
    sg.lbm_nn_status()
    assert torch.equal(dw, want)


def test_conv3_input_gradient_against_oracle():
    """The convolution with the flipped, transposed weights: exact up to FP32 accumulation and one rounding."""
    shape, ci, co = (4, 16, 16), 32, 48
    V = 1024
    rng = np.random.default_rng(0)
    w = rng.standard_normal((co, ci, 3, 3, 3)) * np.sqrt(2.0 / (27 * ci))
    wt = torch.tensor(w.reshape(co, ci, 27), dtype=torch.float32, device="cuda")
    wp = torch.empty(sg.lbm_nn_conv3_packed(co, ci), dtype=torch.bfloat16, device="cuda")
    wtp = torch.empty(sg.lbm_nn_conv3_packed(ci, co), dtype=torch.bfloat16, device="cuda")
    sg.lbm_nn_conv3_pack(wt, wp, wtp, co, ci)
    dy = _rand((V, co), 9)
    dx = torch.empty((V, ci), dtype=torch.bfloat16, device="cuda")
    sg.lbm_nn_conv3((dy, co, 0, None, 0), shape, wtp, ci, dx, ci)
    sg.lbm_nn_status()
    d = np.moveaxis(dy.float().cpu().numpy().reshape(shape + (co,)), -1, 0).astype(np.float64)
    wb = torch.tensor(w).float().to(torch.bfloat16).double().numpy()
    want = orc.conv3d_grad_input(d, wb)
    got = np.moveaxis(dx.float().cpu().numpy().reshape(shape + (ci,)), -1, 0)
    assert np.all(np.abs(got - want) <= 2.0 ** -8 * np.abs(want) + 1e-5)


@pytest.mark.parametrize("C", [8, 16, 48, 160])
@pytest.mark.parametrize("pooled", [False, True])
def test_relu_grad_bias_repeats_the_separate_passes(C, pooled):
    D, H, W = 4, 6, 10
    V = D * H * W
    y, dsk = _rand((V, C), 1), _rand((V, C), 2)
    dy = _rand((V // 8, C), 3) if pooled else _rand((V, C), 3)
    full = dy
    if pooled:
        up = torch.empty((V, C), dtype=torch.bfloat16, device="cuda")
        sg.lbm_nn_pool2(dy, up, D, H, W, C, 1)
        full = torch.empty_like(up)
        sg.lbm_nn_add(up, dsk, full, V * C)
    want = torch.empty((V, C), dtype=torch.bfloat16, device="cuda")
    sg.lbm_nn_relu_grad(y, full, want, V * C)
    got = torch.full((V, C), float("nan"), dtype=torch.bfloat16, device="cuda")
    db = torch.empty(C, dtype=torch.float32, device="cuda")
    sg.lbm_nn_relu_grad_bias(y, dy, dsk if pooled else None, got, db, (D, H, W), C)
    torch.cuda.synchronize()
    assert torch.equal(got, want)
    ref, mag = want.double().sum(0), want.double().abs().sum(0)
    assert torch.all((db.double() - ref).abs() <= V * 2.0 ** -24 * mag + 1e-30)
