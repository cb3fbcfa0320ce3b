"""Convolutions over domains of unusual proportions: more than 65535 planes or tiles along a row."""
import pytest

from tests import test_gpu_conv as conv

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


# a column of 65600 planes, a row of 65600 tiles along x (more than a grid's y or z), both directions' layouts
@pytest.mark.parametrize("shape", [(65600, 2, 4), (2, 2, 524800)])
@pytest.mark.parametrize("ca,up,cb,co", [(5, 0, 0, 16), (16, 0, 0, 16), (16, 1, 16, 32), (160, 0, 0, 16)])
def test_long_domains_repeat_the_gemm(shape, ca, up, cb, co):
    conv.test_conv3_repeats_the_im2col_gemm(shape, ca, up, cb, co)
    conv.test_conv3_wgrad_repeats_the_split_gemm(shape, ca, up, cb, co)
