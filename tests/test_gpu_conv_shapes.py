"""Convolutions over domains of unusual proportions: more than 65535 planes, and planes of more than 2^31 elements."""
import pytest

from tests import test_gpu_conv as conv

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
from paper_2502_12955_gb300 import surrogate as sg  # noqa: E402


# a column of 65600 planes, a row of 65600 tiles along x (more than a grid's y or z), both directions' layouts
@pytest.mark.parametrize("shape", [(65600, 2, 4), (2, 2, 524800)])
@pytest.mark.parametrize("ca,up,cb,co", [(5, 0, 0, 16), (16, 0, 0, 16), (16, 1, 16, 32), (160, 0, 0, 16)])
def test_long_domains_repeat_the_gemm(shape, ca, up, cb, co):
    conv.test_conv3_repeats_the_im2col_gemm(shape, ca, up, cb, co)
    conv.test_conv3_wgrad_repeats_the_split_gemm(shape, ca, up, cb, co)


def test_weight_gradient_with_planes_of_more_than_2_31_elements():
    # values -1, 0, 1: the sums are integers far below 2^24, exact in any order
    D, H, W, C, Co = 2, 8192, 4160, 64, 16
    V = D * H * W
    assert H * W * C >= 1 << 31
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randint(-1, 2, (V, C), generator=g, device="cuda", dtype=torch.int8).to(torch.bfloat16)
    dy = torch.randint(-1, 2, (V, Co), generator=g, device="cuda", dtype=torch.int8).to(torch.bfloat16)
    scratch = torch.empty(sg.lbm_nn_conv3_wgrad_scratch((D, H, W), C, Co), dtype=torch.float32, device="cuda")
    dw = torch.empty((Co, C, 27), dtype=torch.float32, device="cuda")
    sg.lbm_nn_conv3_wgrad((x, C, 0, None, 0), (D, H, W), dy, Co, scratch, dw)
    sg.lbm_nn_status()
    xs, ds = x.view(D, H, W, C), dy.view(D, H, W, Co)
    # taps (dz, dy, dx) that cross the plane in both directions and stay in it
    for dz, ddy, dx in ((1, 0, 0), (-1, 0, 0), (1, -1, 1), (0, 1, 0)):
        want = torch.zeros((Co, C), dtype=torch.float64, device="cuda")
        zd = slice(max(0, -dz), D - max(0, dz))
        for z in range(D)[zd]:
            for y0 in range(0, H, 1024):
                ys = [y for y in (max(y0, -ddy), min(y0 + 1024, H - max(0, ddy)))]
                a = ds[z, ys[0]:ys[1], max(0, -dx):W - max(0, dx)].reshape(-1, Co).float()
                b = xs[z + dz, ys[0] + ddy:ys[1] + ddy, max(0, -dx) + dx:W - max(0, dx) + dx].reshape(-1, C).float()
                want += (a.T @ b).double()
        tap = (dz + 1) * 9 + (ddy + 1) * 3 + dx + 1
        assert torch.equal(dw[:, :, tap].double(), want), (dz, ddy, dx)
