"""The sizes of the GPU tests reach the kernel variants they are there for: what the planner chooses for them, on the host."""
import ctypes

import test_ffn_cluster_shape as FS
import test_gpu_block_strip_loads as S
import test_gpu_pointwise_weights as P
import test_gpu_tile_edges as E
from paper_2212_01005_b200 import binding as B
from paper_2212_01005_b200 import workloads as WL

lib = FS.lib


def cases(test):
    """The parameter sets of a parametrised test."""
    return [m for m in test.pytestmark if m.name == "parametrize"][0].args[1]


# (output rows per strip, shared memory) of the inverted-residual shapes: each is the layout of that many CTAs per strip, and of no
# other number of them but where two are named
SPLITS = {
    (1, 14, 32, 192, 32, 1, True): (1, 34816), (1, 1, 16, 96, 16, 1, True): (1, 24576), (2, 5, 24, 144, 24, 1, True): (1, 44032),      # 6; 3 or 6; 3
    (3, 9, 64, 384, 64, 1, True): (2, 65536), (1, 8, 64, 384, 160, 1, False): (1, 72704), (5, 7, 40, 240, 8, 2, False): (1, 54272),    # 8; 8; 5
    (1, 18, 40, 240, 32, 2, False): (1, 60416), (2, 15, 96, 576, 96, 1, True): (2, 122880), (1, 8, 72, 432, 40, 1, False): (1, 117760),   # 5; 6; 3
    (2, 9, 72, 432, 72, 2, False): (1, 128000), (1, 13, 160, 960, 160, 1, True): (1, 206848), (3, 12, 160, 960, 96, 2, False): (1, 177152),   # 3; 6; 6
    (1, 20, 128, 768, 128, 1, True): (2, 140288), (1, 4, 256, 512, 256, 1, True): (1, 167936),      # 8; 8
    (25, 15, 96, 576, 96, 1, True): (15, 210944), (25, 15, 96, 576, 88, 1, False): (15, 210944),      # 4, 66 KB of sums to exchange: two pieces
    (2, 8, 16, 96, 24, 1, False): (1, 27648), (1, 10, 24, 144, 24, 1, True): (1, 46080), (1, 16, 32, 192, 16, 1, False): (1, 33792),    # 3 or 6; 3; 6
    (9, 22, 16, 96, 16, 1, True): (3, 53248),     # 2
}


def test_inverted_residual_shapes_are_split_over_clusters():
    shapes = cases(E.test_inverted_residual_channel_splits_and_k_blocks)
    assert set(shapes) == set(SPLITS)
    for s in shapes:
        wl = WL.mbv2_block("x", [0], *s)
        sg = B.Subgraph(wl.ops, wl.input_shapes, mode="fused")
        assert (sg.query(B.AGO_Q_TILE_ROWS), sg.query(B.AGO_Q_SMEM_BYTES)) == SPLITS[s], s
        sg.close()


def ffn_plan(lib, rows, d, hidden, d_out):
    q = FS.Shape(M=rows, K=d, Hid=hidden, N2=d_out)
    smem = lib.plan(ctypes.byref(q))
    wl = WL.ffn("x", [0], rows, d, hidden, 1, d_out=d_out)
    sg = B.Subgraph(wl.ops, wl.input_shapes, mode="fused")
    cluster = smem > 0 and sg.query(B.AGO_Q_SMEM_BYTES) == smem and sg.query(B.AGO_Q_TILE_ROWS) == 128
    tile_rows, launches = sg.query(B.AGO_Q_TILE_ROWS), sg.query(B.AGO_Q_NUM_LAUNCHES)
    sg.close()
    return q if cluster else None, tile_rows, launches


def test_feed_forward_shapes_cover_the_variants_of_the_cluster_kernel(lib):
    plans = [ffn_plan(lib, *s) for t in (E.test_feed_forward_splits, E.test_feed_forward_parts_of_several_steps) for s in cases(t)]
    qs = [q for q, _, _ in plans if q]
    assert {q.CS for q in qs} == {2, 3, 4} and {q.BH for q in qs} == {64, 128}
    assert {bool(q.w2_off) for q in qs} == {True, False} and {q.J > 1 for q in qs} == {True, False}
    assert {(q.BH, q.Tp) for q in qs if q.J > 1} >= {(64, 1), (128, 1), (64, 3), (128, 4)}
    assert any(rows == 256 and launches == 2 for q, rows, launches in plans if q is None)      # paired clusters, all blocks split


def test_feed_forward_row_counts_cover_the_rows_kept(lib):
    qs = {rows: ffn_plan(lib, rows, 192, 1024, 512)[0] for rows in cases(E.test_feed_forward_few_rows)}
    assert all(q and q.J > 1 for q in qs.values())
    assert {q.RP for q in qs.values()} >= {16, 32, 64, 80, 128}


def test_feed_forward_staging_shapes_wait_for_the_copies(lib):
    for s in cases(E.test_feed_forward_sums_staged_past_the_ring):
        q = ffn_plan(lib, *s)[0]
        assert q and q.J > 1 and q.wait_copies, s


def test_feed_forward_chains_take_the_kernel_of_the_least_estimate():
    # measured us: pairs / cluster / reduction-tiling kernel, where each was timed
    for shape, (tile_rows, smem) in {(4157, 128, 2048, 256): (128, 230912),      # cluster: 41 / 32 / -
                                     (646, 64, 3328, 384): (128, 165120),       # reduction: - / 38 / 25
                                     (2500, 768, 3072, 768): (256, 214528),     # pairs: 50 / 67 / -
                                     (12288, 768, 3072, 768): (256, 214528)}.items():
        wl = WL.ffn("x", [0], *shape[:3], 1, d_out=shape[3])
        sg = B.Subgraph(wl.ops, wl.input_shapes, mode="fused")
        assert (sg.query(B.AGO_Q_TILE_ROWS), sg.query(B.AGO_Q_SMEM_BYTES)) == (tile_rows, smem), shape
        sg.close()


def variant(wl):
    sg = B.Subgraph(wl.ops, wl.input_shapes, mode="fused")
    v = sg.query(B.AGO_Q_FUSED_VARIANT)
    sg.close()
    return v


# Shapes whose strip and first weights the threads copy: the others of the two tests take them by TMA. (bytes of the strip, its pixels)
COPIED_STRIPS = {
    (40, 7, 7, 32, 192, 32, 1, True), (1, 33, 31, 32, 96, 16, 1, False), (1, 32, 32, 32, 96, 16, 1, False),      # 4032 to 6144 bytes
    (9, 12, 10, 256, 512, 64, 1, False),      # 30720 bytes, 60 pixels (68 and 75 go by TMA)
    (8, 28, 28, 16, 96, 24, 1, False),      # 17920 bytes, pixels of 32
    (30, 13, 9, 72, 144, 24, 2, False), (12, 14, 14, 136, 768, 136, 1, True), (2, 24, 168, 64, 1),      # pixels that end inside a sector
    (4, 20, 32, 128, 1), (3, 31, 64, 96, 2),      # 6400 and 11904 bytes (13056 go by TMA)
}


def test_inverted_residual_strips_come_as_their_rule_says():
    blocks, pairs = cases(S.test_block), cases(S.test_pointwise_depthwise)
    assert COPIED_STRIPS <= set(blocks) | set(pairs)
    for s in blocks:
        assert variant(S.block(s)) == (s not in COPIED_STRIPS), s
    for s in pairs:
        assert variant(WL.pw_dw("x", [0], *s)) == (s not in COPIED_STRIPS), s
    assert variant(WL.dw_pw("x", [0], 32, 28, 96, 32, 1)) == 0


# Shapes whose weights the threads copy. (CTAs, bytes of weights)
COPIED_WEIGHTS = {
    (1, 36, 48, 24, 48), (1, 46, 144, 24, 144),      # pairs: 41 CTAs (40 take them by TMA); 67 CTAs, 13824 bytes (64 by TMA, and 72 with 30720 bytes)
    (2, 70, 96, 32, 96),      # 148 CTAs, 12288 bytes in whole rows, tiles of 67 rows (of 64 go by TMA)
    (1, 4, 320, 32, 32, 64), (1, 4, 324, 32, 32, 64), (1, 4, 196, 48, 48, 96),      # chains: 25 to 41 CTAs, 6144 and 13824 bytes (24 CTAs by TMA)
    (1, 4, 584, 120, 120, 240), (3, 4, 196, 120, 120, 240),      # 73 and 74 CTAs, rows that end inside 64 bytes (72 by TMA)
    (1, 1, 1, 8, 8, 8),      # a chain's weights in rows of 16 bytes
    (32, 4, 284, 96, 96, 192),      # one CTA per SM, whole rows, tiles of 123 rows (of 111 by TMA)
}


def test_pointwise_weights_come_as_their_rule_says():
    pairs, chains = cases(P.test_pointwise_pair), cases(P.test_unfold_chain)
    assert COPIED_WEIGHTS <= set(pairs) | set(chains)
    for s in pairs:
        assert variant(P.pair(s)) == (s not in COPIED_WEIGHTS), s
    for s in chains:
        assert variant(P.chain(s)) == (s not in COPIED_WEIGHTS), s


def test_feed_forward_variants_are_named():
    for (rows, d, hidden, d_out), v in {(646, 64, 3328, 384): 0, (12288, 64, 256, 128): 1, (512, 768, 3072, 768): 2, (12288, 768, 3072, 768): 3}.items():
        assert variant(WL.ffn("x", [0], rows, d, hidden, 1, d_out=d_out)) == v
    wl = WL.get("ffn_512")
    sg = B.Subgraph(wl.ops, wl.input_shapes, mode="per_mini_subgraph")
    assert sg.query(B.AGO_Q_FUSED_VARIANT) == 0
    sg.close()
