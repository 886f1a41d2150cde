"""Inverted-residual blocks whose input strip and W1 come by TMA, on both sides of that rule (which shape takes which is checked on the
host, test_tilings.py) and at the edges of its loads (several K blocks, the last one part empty, W1 in several loads, first and last
strips, strips past the image), against the oracle. Tolerance: the one of the parity tests (bf16 in and out, fp32 accumulate: max|gpu - ref| <= 1e-2 max|ref| + 1e-3)."""
import pytest

from paper_2212_01005_b200 import workloads as WL
from test_gpu_tile_edges import check

pytestmark = pytest.mark.gpu


def block(shape):
    n, h, w, cin, cexp, cout, stride, residual = shape
    return WL.Workload("block_strips", [240, *shape[:7]], [(n, h, w, cin)], WL._mbv2_ops(cexp, cout, stride, residual), samples=n, input_dist=["uniform"])


@pytest.mark.parametrize("shape", [
    # n, h, w, c_in, c_exp, c_out, stride, residual
    (40, 7, 7, 32, 192, 32, 1, True), (1, 33, 31, 32, 96, 16, 1, False), (1, 32, 32, 32, 96, 16, 1, False), (1, 3, 120, 64, 128, 64, 1, True),
    (30, 13, 9, 72, 144, 24, 2, False), (25, 15, 15, 96, 576, 96, 1, True), (12, 14, 14, 136, 768, 136, 1, True), (3, 29, 27, 64, 384, 64, 1, True),
    (160, 14, 14, 32, 512, 32, 1, True), (32, 28, 28, 32, 192, 64, 2, False), (2, 57, 58, 32, 192, 40, 2, False), (6, 20, 20, 64, 384, 160, 1, False),
    (9, 12, 10, 256, 512, 64, 1, False), (26, 8, 8, 160, 960, 96, 1, False), (4, 15, 15, 96, 576, 96, 2, False),
    (8, 28, 28, 16, 96, 24, 1, False), (4, 16, 15, 112, 160, 112, 1, True), (5, 14, 17, 120, 192, 48, 2, False), (2, 9, 23, 168, 64, 24, 1, False),
])
def test_block(ago, shape):
    check(ago, block(shape))


@pytest.mark.parametrize("shape", [(4, 20, 32, 128, 1), (3, 31, 64, 96, 2), (2, 17, 96, 192, 1), (2, 24, 168, 64, 1), (1, 26, 120, 48, 1)])      # n, h, c_in, c_exp, stride
def test_pointwise_depthwise(ago, shape):
    check(ago, WL.pw_dw("pw_dw_strips", [241, *shape], *shape))
