"""Pointwise pairs and unfolded projection chains whose weights come by TMA, on both sides of that rule (which shape takes which is
checked on the host, test_tilings.py) and at the edges of its loads (padded channels, several blocks, blocks of more than 256 rows),
against the oracle. Tolerance: the one of the parity tests (bf16 in and out, fp32 accumulate: max|gpu - ref| <= 1e-2 max|ref| + 1e-3)."""
import pytest

from paper_2212_01005_b200 import workloads as WL
from test_gpu_tile_edges import check

pytestmark = pytest.mark.gpu


def pair(shape):
    n, h, c0, c1, c2 = shape
    return WL.pw_pw("pw_pw_weights", [230, *shape], n, h, c0, c1, c2)


def chain(shape):
    b, p, n, c0, c1, c2 = shape
    m = b * p * n
    ops = [("gemm", dict(N=c1)), ("reshape", dict(shape=(b * p, n, c1))), ("add_input", dict(input=1)),
           ("reshape", dict(shape=(b, p, n, c1))), ("transpose", dict(a=1, b=2)), ("reshape", dict(shape=(m, c1))),
           ("gemm", dict(N=c2)), ("reshape", dict(shape=(b, n, p, c2)))]
    return WL.Workload("unfold_weights", [231, *shape], [(m, c0), (b * p, n, c1)], ops, samples=b, input_dist=["normal", "normal"])


@pytest.mark.parametrize("shape", [
    # n, h, c0, c1, c2: one pixel; one CTA; 40 and 41 CTAs of 32 rows; 72 with 30 KB of weights, 64 and 67 with 13.8 KB; 148 with rows of 64 bytes
    (1, 1, 8, 8, 8), (1, 5, 24, 8, 40), (1, 7, 200, 120, 104), (5, 16, 48, 24, 48), (1, 36, 48, 24, 48),
    (9, 16, 192, 40, 192), (1, 48, 192, 40, 192), (1, 97, 192, 32, 192), (2, 70, 96, 32, 96), (1, 20, 264, 72, 136),
    (2, 32, 144, 24, 144), (1, 46, 144, 24, 144),
])
def test_pointwise_pair(ago, shape):
    check(ago, pair(shape))


@pytest.mark.parametrize("shape", [
    # images, pixels per patch, patches, C0, C1, C2: one row per image; blocks of 264, 320 and 512 rows; 40 and 41 CTAs; 148 with whole rows;
    # 24 and 25 CTAs with 13.8 KB of weights, 72 and 73 with 86 KB; tiles of 111 and 123 rows
    (1, 1, 1, 8, 8, 8), (1, 1, 1, 16, 16, 16), (1, 4, 9, 264, 40, 64), (2, 4, 16, 320, 64, 128), (1, 4, 25, 512, 24, 72), (1, 4, 320, 32, 32, 64),
    (1, 4, 324, 32, 32, 64), (6, 4, 196, 64, 64, 128), (9, 9, 256, 96, 96, 192), (3, 4, 196, 120, 120, 240),
    (1, 4, 192, 48, 48, 96), (1, 4, 196, 48, 48, 96), (1, 4, 576, 120, 120, 240), (1, 4, 584, 120, 120, 240), (32, 4, 256, 96, 96, 192), (32, 4, 284, 96, 96, 192),
])
def test_unfold_chain(ago, shape):
    check(ago, chain(shape))
