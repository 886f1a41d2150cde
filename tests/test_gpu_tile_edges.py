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


@pytest.mark.parametrize("shape", [
    # n, h, c_in, c_exp, c_out, stride, residual: channels split over clusters of 2 to 8 CTAs
    (1, 14, 32, 192, 32, 1, True), (1, 1, 16, 96, 16, 1, True), (2, 5, 24, 144, 24, 1, True), (3, 9, 64, 384, 64, 1, True),
    (1, 8, 64, 384, 160, 1, False), (5, 7, 40, 240, 8, 2, False), (1, 18, 40, 240, 32, 2, False),
    # more than 64 input channels: two and three K blocks, whole and with a remainder of one or more steps, padded last step
    (2, 15, 96, 576, 96, 1, True), (1, 8, 72, 432, 40, 1, False), (2, 9, 72, 432, 72, 2, False), (1, 13, 160, 960, 160, 1, True),
    (3, 12, 160, 960, 96, 2, False), (1, 20, 128, 768, 128, 1, True), (1, 4, 256, 512, 256, 1, True),
    # partial sums exchanged in two pieces, the second one as wide as the first and narrower
    (25, 15, 96, 576, 96, 1, True), (25, 15, 96, 576, 88, 1, False),
    # widths that cut into one, two, three odd segments with and without a remainder; rows that leave half a block
    (2, 8, 16, 96, 24, 1, False), (1, 10, 24, 144, 24, 1, True), (1, 16, 32, 192, 16, 1, False), (9, 22, 16, 96, 16, 1, True),
])
def test_inverted_residual_channel_splits_and_k_blocks(ago, shape):
    n, h, c_in, c_exp, c_out, stride, residual = shape
    check(ago, WL.mbv2_block("mbv2_edges", [202, *map(int, shape)], n, h, c_in, c_exp, c_out, stride, residual))


@pytest.mark.parametrize("shape, rows, smem", [
    # n, h, c, c_exp: two, three and four K blocks, with and without a remainder; strips of several rows and of one
    ((64, 15, 80, 240), 8, 217088), ((64, 14, 96, 192), 7, 166912), ((25, 14, 88, 176), 3, 150528), ((3, 9, 72, 16), 1, 58368),
    ((40, 9, 144, 48), 3, 113664), ((20, 12, 136, 32), 2, 91136), ((2, 7, 200, 16), 1, 99328), ((1, 5, 256, 16), 1, 99328),
])
def test_wide_residual_blocks_that_are_not_split(ago, shape, rows, smem):
    # the residual comes from the K blocks of the input tile; the tiling is the unsplit one of these strips
    n, h, c, c_exp = shape
    wl = WL.mbv2_block("mbv2_wide", [214, *shape], n, h, c, c_exp, c, 1, True)
    sg = ago.Subgraph(wl.ops, wl.input_shapes, mode="fused")
    assert (sg.query(ago.AGO_Q_TILE_ROWS), sg.query(ago.AGO_Q_SMEM_BYTES)) == (rows, smem)
    sg.close()
    check(ago, wl)


def test_split_channels_repeat_within_the_order_of_the_groups(ago):
    # many launches in flight on clusters that share SMs with the next grid's: every result stays that of the first one, up to
    # the order in which the groups add their chunks (one bf16 step)
    import torch
    from helpers import to_device
    wl = WL.mbv2_block("mbv2_repeat", [203], 25, 15, 96, 576, 96, 1, True)
    data = WL.generate(wl)
    sg = ago.Subgraph(wl.ops, wl.input_shapes, mode="fused")
    ins, ws = to_device(wl, data)
    outs = [sg.run(ins, ws) for _ in range(40)]
    torch.cuda.synchronize()
    assert sg.status() == ago.AGO_OK, ago.ago_last_error()
    scale = float(outs[0].float().abs().max())
    for o in outs[1:]:
        assert float((o.float() - outs[0].float()).abs().max()) <= 2.0 ** -7 * scale
    sg.close()


@pytest.mark.parametrize("rows", [1, 15, 16, 17, 63, 64, 65, 127, 128, 129, 256, 257, 513])
def test_feed_forward_few_rows(ago, rows):
    # rows kept in shared memory (16 .. 128), direct and staged additions (64 rows), one to five row blocks; hidden tiles of 64
    check(ago, WL.ffn("ffn_rows", [204, rows], rows, 192, 1024, 1, d_out=512))


@pytest.mark.parametrize("shape", [
    # rows, d, hidden, d_out: the second GEMM's tiles behind the ring and in stages of their own, clusters of 2, 3 and 4, one and
    # more steps per cluster, tiles of 64 and of 128; whole row blocks without a split (24 blocks); paired clusters all split
    (40, 64, 256, 128), (100, 256, 768, 192), (100, 1024, 4096, 1024), (200, 128, 384, 768), (300, 64, 2048, 256),
    (700, 320, 1536, 384), (1500, 128, 768, 512), (3001, 128, 512, 256), (2500, 192, 3072, 768),
])
def test_feed_forward_splits(ago, shape):
    rows, d, hidden, d_out = shape
    check(ago, WL.ffn("ffn_splits", [205, *shape], rows, d, hidden, 1, d_out=d_out))


def test_feed_forward_few_rows_leave_the_sums_clean(ago):
    # the fp32 buffer of the split row blocks is zeroed by the run itself: many runs in flight agree with the first one
    import torch
    from helpers import to_device
    wl = WL.ffn("ffn_clean", [206], 40, 256, 1024, 1)
    data = WL.generate(wl)
    sg = ago.Subgraph(wl.ops, wl.input_shapes, mode="fused")
    ins, ws = to_device(wl, data)
    outs = [sg.run(ins, ws) for _ in range(20)]
    torch.cuda.synchronize()
    assert sg.status() == ago.AGO_OK, ago.ago_last_error()
    scale = float(outs[0].float().abs().max())
    for o in outs[1:]:
        assert float((o.float() - outs[0].float()).abs().max()) <= 2.0 ** -7 * scale     # one bf16 step: the order of the additions
    sg.close()


@pytest.mark.parametrize("shape", [(646, 64, 3328, 384), (1000, 64, 3328, 384), (1500, 128, 2432, 256)])
def test_feed_forward_uneven_splits_on_the_reduction_kernel(ago, shape):
    # hidden tiles (26, 19) that the row blocks' clusters cannot share out evenly
    rows, d, hidden, d_out = shape
    wl = WL.ffn("ffn_uneven", [222, *shape], rows, d, hidden, 1, d_out=d_out)
    sg = ago.Subgraph(wl.ops, wl.input_shapes, mode="fused")
    assert sg.query(ago.AGO_Q_NUM_LAUNCHES) == 1 and sg.query(ago.AGO_Q_SMEM_BYTES) == 165120
    sg.close()
    check(ago, wl)


@pytest.mark.parametrize("shape", [(2025, 128, 1536, 512), (1632, 64, 3072, 384)])
def test_feed_forward_parts_of_several_steps(ago, shape):
    # split row blocks whose parts take three steps of tiles of 64 and four of 128: the ring goes round, sums staged over it at the end
    rows, d, hidden, d_out = shape
    check(ago, WL.ffn("ffn_parts", [221, *shape], rows, d, hidden, 1, d_out=d_out))


@pytest.mark.parametrize("shape", [(300, 64, 2048, 256), (1000, 128, 512, 384), (128, 256, 3072, 768), (65, 64, 1024, 256)])
def test_feed_forward_sums_staged_past_the_ring(ago, shape):
    # narrow inputs, wide outputs: the staged sums reach the hidden tiles' slots. Many launches in flight, each against the oracle.
    import torch
    from helpers import to_device
    rows, d, hidden, d_out = shape
    wl = WL.ffn("ffn_staging", [217, *shape], rows, d, hidden, 1, d_out=d_out)
    data = WL.generate(wl)
    ref = O.run_chain(wl.ops, data["inputs"], data["weights"])
    sg = ago.Subgraph(wl.ops, wl.input_shapes, mode="fused")
    assert sg.query(ago.AGO_Q_NUM_LAUNCHES) == 2         # split row blocks
    ins, ws = to_device(wl, data)
    outs = [sg.run(ins, ws) for _ in range(100)]
    torch.cuda.synchronize()
    assert sg.status() == ago.AGO_OK, ago.ago_last_error()
    for o in outs:
        assert_close(o.double().cpu().numpy(), ref, what=f"ffn {shape}")
    sg.close()


@pytest.mark.parametrize("shape", [
    # rows, K, N of one GEMM + bias + GELU: tiles of 128 x 64 (few tiles; N a remainder of 64), 128 x 128, pairs with tiles of 256
    # and of 128 columns (N a remainder of either), more K blocks than ring stages and fewer
    (70, 72, 40), (130, 1024, 72), (500, 640, 136), (600, 64, 2056), (2100, 768, 200), (3001, 200, 776), (4097, 64, 1032), (19000, 96, 264),
])
def test_unfused_gemm_tiles(ago, shape):
    rows, k, n = shape
    ops = [("gemm", dict(N=n)), ("bias_add", {}), ("gelu_tanh", {})]
    check(ago, WL.Workload("gemm_tiles", [207, *shape], [(rows, k)], ops, samples=1), mode="per_mini_subgraph")


@pytest.mark.parametrize("shape", [
    # pixels, c_in, c_mid, c_out: one tile of 32 rows per SM and around it, of 128 rows, two CTAs per SM, two rounds
    (1, 64, 32, 64), (32, 96, 24, 96), (33, 8, 8, 8), (4736, 64, 32, 64), (4737, 64, 24, 72), (18944, 64, 32, 64), (18945, 72, 24, 64),
    (37889, 48, 16, 48),
    # two rounds with one CTA per SM; with two CTAs per SM whose products share their columns; padding in every operand
    (18945, 256, 64, 256), (37889, 64, 64, 256), (40000, 24, 40, 88),
])
def test_pointwise_pair_tiles(ago, shape):
    m, c0, c1, c2 = shape
    check(ago, WL.pw_pw("pw_pw_edges", [207, *shape], m, 1, c0, c1, c2, act1=True))


@pytest.mark.parametrize("shape", [(2, 20, 264, 24, 64), (3, 14, 320, 40, 160), (20, 14, 512, 8, 24), (1, 9, 272, 120, 72)])
def test_pointwise_pair_padding_over_wide_inputs(ago, shape):
    # middle widths padded by eight rows of weights whose 16-byte pieces are more than the threads that clear them; shared memory
    # holds NaN from the launch before (the input tile of 512 channels covers the first 128 KB on every SM)
    import torch
    n, h, c0, c1, c2 = shape
    fill = WL.Workload("pw_pw_fill", [215], [(148, 128, 1, 512)], WL.pw_pw("x", [0], 1, 1, 512, 64, 64).ops, samples=148)
    sg = ago.Subgraph(fill.ops, fill.input_shapes, mode="fused")
    assert sg.query(ago.AGO_Q_SMEM_BYTES) > 128 * 1024
    nan = [torch.full(s, float("nan"), dtype=torch.float32 if k == "bias" else torch.bfloat16, device="cuda")
           for s, k in zip(fill.input_shapes + fill.weight_shapes, ["input"] + fill.weight_kinds)]
    sg.run(nan[:1], nan[1:])
    torch.cuda.synchronize()
    check(ago, WL.pw_pw("pw_pw_padding", [216, *shape], n, h, c0, c1, c2))
    sg.close()


@pytest.mark.parametrize("shape", [(5, 9, 421, 96, 192), (3, 4, 3200, 64, 256), (1, 9, 2113, 40, 24)])
def test_unfold_chain_rounds(ago, shape):
    check(ago, WL.unfold_chain("unfold_edges", [208, *shape], *shape))


def test_pointwise_pair_output_between_sectors(ago):
    # an output 16 but not 32 bytes aligned: rows are stored in halves
    import torch
    from helpers import to_device
    wl = WL.pw_pw("pw_pw_offset", [209], 3, 20, 64, 32, 64)
    data = WL.generate(wl)
    sg = ago.Subgraph(wl.ops, wl.input_shapes, mode="fused")
    ins, ws = to_device(wl, data)
    ref = sg.run(ins, ws)
    flat = torch.zeros(ref.numel() + 16, dtype=ref.dtype, device=ref.device)
    out = flat[8:8 + ref.numel()].view(ref.shape)
    sg.run(ins, ws, out=out)
    torch.cuda.synchronize()
    assert sg.status() == ago.AGO_OK and torch.equal(out, ref)
    assert not flat[:8].any() and not flat[-8:].any()
    sg.close()


BETWEEN_SECTORS = [
    # paired clusters, blocks in the middle of a cluster's run and its last one; a cluster with whole row blocks
    (WL.ffn("ffn_offset", [242], 17000, 64, 256, 1, d_out=768), "fused", 3), (WL.ffn("ffn_offset", [243], 12300, 64, 256, 1, d_out=128), "fused", 1),
    # 64 channels in two column phases, whose residual is read by whole sectors where it starts on one: the pair, and the single
    # convolution of the unfused mode with the residual in its epilogue; one phase
    (WL.Workload("conv_offset", [244], [(14, 35, 33, 64)], WL.resnet_block("x", [0], 1, 8, 64).ops, samples=14, input_dist=["relu_normal"]), "fused", 0),
    (WL.Workload("conv_offset", [245], [(14, 35, 33, 64)], WL.resnet_block("x", [0], 1, 8, 64).ops, samples=14, input_dist=["relu_normal"]), "per_mini_subgraph", 0),
    (WL.Workload("conv_offset", [246], [(2, 9, 9, 32)], WL.resnet_block("x", [0], 1, 8, 32).ops, samples=2, input_dist=["relu_normal"]), "fused", 0),
]


@pytest.mark.parametrize("wl, mode, variant", BETWEEN_SECTORS, ids=["ffn_pair", "ffn_cluster", "conv_pair", "conv_single", "conv_one_phase"])
def test_tensors_between_sectors(ago, wl, mode, variant):
    # inputs and output 16 but not 32 bytes aligned take other loads and stores than aligned ones, for the same values
    import torch
    from helpers import to_device
    sg = ago.Subgraph(wl.ops, wl.input_shapes, mode=mode)
    assert sg.query(ago.AGO_Q_FUSED_VARIANT) == variant
    ins, ws = to_device(wl, WL.generate(wl))

    def shifted(t):      # the tensor 16 bytes into a buffer with a guard on either side
        flat = torch.zeros(t.numel() + 16, dtype=t.dtype, device=t.device)
        flat[8:8 + t.numel()] = t.flatten()
        return flat, flat[8:8 + t.numel()].view(t.shape)

    ref = sg.run(ins, ws)
    flat, out = shifted(torch.full_like(ref, float("nan")))
    moved = [shifted(t)[1] for t in ins]
    assert all(t.data_ptr() % 32 == 16 for t in moved + [out])
    sg.run(moved, ws, out=out)
    only_out = torch.empty_like(ref)
    sg.run(moved, ws, out=only_out)
    torch.cuda.synchronize()
    assert sg.status() == ago.AGO_OK and torch.equal(out, ref) and torch.equal(only_out, ref)
    assert not flat[:8].any() and not flat[-8:].any()
    sg.close()
    if ref.numel() < 2000000:
        check(ago, wl, mode)


@pytest.mark.parametrize("fp32", [True, False])
@pytest.mark.parametrize("shape", [
    # n, h, w, c, stride: one pixel, one row, one column, fewer pixels than a piece; even and odd sizes at stride 2
    (1, 1, 1, 8, 1), (1, 1, 9, 16, 2), (3, 7, 1, 8, 1), (1, 3, 2, 24, 2), (2, 6, 5, 8, 1),
    # two rows by two and by four columns, four rows by four and by eight, each with ragged last pieces
    (5, 27, 13, 56, 1), (19, 23, 23, 64, 1), (23, 29, 21, 88, 1), (21, 45, 37, 144, 1),
    (19, 29, 27, 96, 2), (9, 53, 51, 128, 2), (13, 73, 67, 144, 2), (15, 93, 91, 176, 2),
])
def test_depthwise_strips(ago, shape, fp32):
    n, h, w, c, stride = shape
    ops = [("conv2d", dict(O=c, R=3, S=3, stride=stride, pad=1, groups=c)), ("bias_add", {}), ("relu6", {})]
    wl = WL.Workload("dw_edges", [210, *shape], [(n, h, w, c)], ops, samples=n, input_dist=["normal"])
    data = WL.generate(wl)
    ref = O.run_chain(wl.ops, data["inputs"], data["weights"])
    out = run_gpu(ago, wl, data, "auto", fp32=fp32)
    if fp32:   # nine products and a bias, each sum rounded: 10 x 2^-24 of the sum of the magnitudes, itself below 9 x 5 max
        assert abs(out - ref).max() <= 1e-5 * max(1.0, abs(ref).max())
    else:
        assert_close(out, ref, what=f"depthwise {shape}")


@pytest.mark.parametrize("ops", [
    [], [("relu", {})], [("bias_add", {})], [("bias_add", {}), ("relu", {})], [("bias_add", {}), ("gelu_tanh", {})],
    [("scale", dict(f=0.5)), ("bias_add", {}), ("relu6", {})], [("bias_add", {}), ("add_input", dict(input=0)), ("relu", {})],
])
def test_depthwise_strips_epilogues(ago, ops):
    wl = WL.Workload("dw_epilogues", [211], [(3, 22, 19, 40)], [("conv2d", dict(O=40, R=3, S=3, stride=1, pad=1, groups=40))] + ops,
                     samples=3, input_dist=["normal"])
    check(ago, wl, "auto")


@pytest.mark.parametrize("shape", [
    # n, h, w, c: one pixel, one row, one column; a tile and a position more; one and two column phases
    (1, 1, 1, 16), (2, 1, 9, 32), (1, 9, 1, 64), (1, 3, 2, 16), (2, 15, 16, 64), (1, 7, 14, 64), (3, 8, 29, 32),
    (14, 35, 33, 64), (4, 41, 42, 16), (33, 56, 54, 64), (13, 61, 59, 32), (20, 57, 75, 16), (5, 78, 76, 64),
    # rows wider than one box: pieces of 32 positions
    (1, 5, 253, 16), (1, 4, 300, 16), (1, 3, 560, 32), (2, 2, 896, 16),
])
def test_residual_block_phases_and_tiles(ago, shape):
    n, h, w, c = shape
    ops = WL.resnet_block("x", [0], 1, 8, c).ops
    check(ago, WL.Workload("residual_edges", [212, *shape], [shape], ops, samples=n, input_dist=["relu_normal"]))


@pytest.mark.parametrize("shape", [(1, 1, 1, 16), (2, 9, 31, 64), (30, 56, 55, 64), (6, 40, 254, 16), (17, 33, 30, 32)])
def test_single_convolution_phases_and_tiles(ago, shape):
    n, h, w, c = shape
    ops = [("conv2d", dict(O=c, R=3, S=3, stride=1, pad=1, groups=1)), ("bias_add", {}), ("relu", {})]
    check(ago, WL.Workload("conv_edges", [213, *shape], [shape], ops, samples=n, input_dist=["relu_normal"]), "per_mini_subgraph")


@pytest.mark.parametrize("seq", [200, 384])
def test_attention_outlier_in_a_middle_chunk(ago, seq):
    # one key far above the 32 that give every row its reference value, in a middle chunk of 32 keys of a half (head 0: first half,
    # head 1: second): its probability is one, whichever pipe evaluates the exponential. One image per place in the chunk and gap in
    # nats: below, around and far beyond where 2^x leaves the exponent field.
    import numpy as np
    cases = [(gap, place) for gap in (60.0, 90.0, 120.0, 208.0, 300.0) for place in range(32)]
    half = 112 if seq == 200 else 192
    wl = WL.attention("attn_outlier", [218, seq], len(cases), seq, 2, 64)
    rng = np.random.default_rng([218, seq])
    q, k = np.zeros(wl.input_shapes[0], np.float32), rng.uniform(-1, 1, wl.input_shapes[0]).astype(np.float32)
    v = rng.uniform(-1, 1, wl.input_shapes[0]).astype(np.float32)
    for b, (gap, place) in enumerate(cases):
        for head, key in enumerate((64 + place, half + (64 if seq == 384 else 32) + place)):
            k[b, :, head * 64] = 0.0
            k[b, key, head * 64] = 32.0
            q[b, :, head * 64] = gap / 4.0          # 32 * gap / 4 / sqrt(64) = gap
            q[b, :, head * 64 + 32:head * 64 + 64] = 0.5
    data = {"inputs": [WL.bf16_round(a) for a in (q, k, v)], "weights": []}
    ref = O.run_chain(wl.ops, data["inputs"], [])
    assert_close(run_gpu(ago, wl, data, "fused"), ref, what=f"attention outlier S={seq}")


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_attention_rows_with_a_non_finite_score_are_nan(ago, value):
    # one key of an image scores NaN or +inf for every query: softmax has no finite value, whichever place of a chunk it is at (first,
    # third and last chunk of a half)
    import torch
    keys = list(range(32)) + list(range(64, 96)) + list(range(160, 192))
    wl = WL.attention("attn_nan", [219], len(keys), 384, 1, 64)
    g = torch.Generator(device="cuda").manual_seed(219)
    q, k, v = (torch.rand(wl.input_shapes[0], generator=g, device="cuda").add_(0.1).to(torch.bfloat16) for _ in range(3))
    for b, key in enumerate(keys):
        k[b, key, 0] = value
    sg = ago.Subgraph(wl.ops, wl.input_shapes, mode="fused")
    out = sg.run([q, k, v], [])
    torch.cuda.synchronize()
    assert sg.status() == ago.AGO_OK, ago.ago_last_error()
    assert out.isnan().all(), [keys[b] for b in range(len(keys)) if not bool(out[b].isnan().all())]
    sg.close()


@pytest.mark.parametrize("mode", ["fused", "per_mini_subgraph"])
@pytest.mark.parametrize("shape, value", [((1, 9, 9, 16), float("nan")), ((4, 30, 33, 64), float("nan")), ((2, 12, 12, 32), float("inf"))])
def test_residual_block_relu_of_a_nan_is_zero(ago, shape, value, mode):
    # one non-finite input value: the sums over it are NaN or infinite; ReLU makes 0 of a NaN in every kernel, as in the oracle
    import numpy as np
    wl = WL.Workload("residual_nan", [220, *shape], [shape], WL.resnet_block("x", [0], 1, 8, shape[3]).ops, samples=shape[0], input_dist=["relu_normal"])
    data = WL.generate(wl)
    data["inputs"][0][0, 4, 4, 3] = value
    ref = O.run_chain(wl.ops, data["inputs"], data["weights"])
    out = run_gpu(ago, wl, data, mode)
    assert np.array_equal(np.isfinite(out), np.isfinite(ref)) and not np.isnan(out).any()
    finite = np.isfinite(ref)
    assert_close(out[finite], ref[finite], what=f"residual with {value} {mode}")


@pytest.mark.parametrize("mode", ["per_mini_subgraph", "per_op"])
@pytest.mark.parametrize("shape", [
    # rows, d, hidden, d_out on pairs of CTAs: last tiles of 8, 72, 104 and 232 columns and of 1, 44 and 196 rows; reductions that end
    # inside a block; weights whose columns are whole blocks of 64 (one load for all) and not; one to three tiles per pair
    (1100, 72, 2056, 136), (2500, 200, 1000, 968), (9473, 64, 264, 104), (5120, 128, 1024, 512), (8001, 40, 1088, 256),
])
def test_paired_gemm_edges(ago, shape, mode):
    rows, d, hidden, d_out = shape
    check(ago, WL.ffn("gemm_pair_edges", [230, *shape], rows, d, hidden, 1, d_out=d_out), mode)


@pytest.mark.parametrize("shape", [
    # 256-row blocks on paired clusters: one, three and five K blocks (an odd one leaves half a pair of stages empty), 256 to 768
    # outputs (the halves of the chunks side by side), whole blocks before split ones, several blocks per cluster
    (7200, 64, 256, 256), (7000, 192, 512, 768), (8700, 320, 512, 512), (17000, 64, 256, 768), (9000, 128, 768, 768),
])
def test_feed_forward_paired_clusters(ago, shape):
    rows, d, hidden, d_out = shape
    check(ago, WL.ffn("ffn_pair_edges", [231, *shape], rows, d, hidden, 1, d_out=d_out))
