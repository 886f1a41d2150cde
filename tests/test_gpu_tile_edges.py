"""Kernel variants at the sizes where their tiles, segments and remainders change, against the oracle. Tolerance: the one
of the parity tests (bf16 in and out, fp32 accumulate: max|gpu - ref| <= 1e-2 max|ref| + 1e-3)."""
import pytest

from oracle import oracle as O
from paper_2212_01005_b200 import workloads as WL
from helpers import assert_close, run_gpu

pytestmark = pytest.mark.gpu


def check(ago, wl, mode="fused"):
    data = WL.generate(wl)
    ref = O.run_chain(wl.ops, data["inputs"], data["weights"])
    assert_close(run_gpu(ago, wl, data, mode), ref, what=f"{wl.name} {wl.input_shapes} {mode}")


@pytest.mark.parametrize("shape", [
    (1, 1, 1, 16), (2, 2, 1, 16), (1, 1, 9, 32), (1, 5, 2, 48),      # one row, one column, fewer columns than a halo
    (1, 6, 4, 16), (1, 6, 5, 16), (3, 9, 7, 16), (2, 9, 8, 80),      # one segment, one segment and one column (4 and 7 columns)
    (1, 20, 15, 144), (2, 31, 22, 16), (4, 64, 57, 48),              # ragged last segments and strips, many strips
])
def test_depthwise_pair_segments_and_strips(ago, shape):
    c = shape[3]
    check(ago, WL.Workload("dw_dw_edges", [201, *shape], [shape], WL.dw_dw("x", [0], 1, 8, c).ops, samples=shape[0], input_dist=["relu_normal"]))
