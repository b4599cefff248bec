"""Choices of lc_variant_default that measured slower when made otherwise (no GPU needed: the plans
a default descriptor resolves to)."""

import pytest

from paper_1405_7470_gb300 import lc


@pytest.fixture(scope="module")
def kernel():
    from paper_1405_7470_gb300 import build
    build()
    return lc.Kernel()


def default(kernel, E, N, F, layout, precision):
    v = lc.variant_default(kernel, E, N, F, layout, precision)
    return v, lc.variant_plan(kernel, E, N, F, v)


@pytest.mark.parametrize("layout", ["elem", "node"])
@pytest.mark.parametrize("N,F,E", [(20, 4, 187501), (20, 4, 40000), (32, 3, 97657), (24, 3, 173611), (28, 3, 35714),
                                   (20, 1, 4096), (48, 1, 200000), (84, 2, 20000)])
def test_fp64_blocks_of_even_width(kernel, layout, N, F, E):
    """The columns of all blocks together, padding included, stay within a quarter of F N."""
    v, p = default(kernel, E, N, F, layout, "fp64")
    width = p["threads"] // (v.tile_e // v.elems_per_thread) * v.split_i
    assert p["column_blocks"] * width <= 1.25 * F * N


def test_fp64_small_batch_keeps_small_tiles(kernel):
    v, _ = default(kernel, 4096, 20, 1, "elem", "fp64")
    assert (v.elems_per_thread, v.split_i, v.tile_e) == (2, 2, 32)


@pytest.mark.parametrize("layout,N,F,E,want", [
    ("node", 4, 6, 357140, (8, 4, 128, 4)), ("node", 6, 8, 46296, (8, 4, 128, 4)), ("node", 4, 6, 357141, (4, 8, 64, 4)),
    ("node", 10, 8, 111108, (4, 8, 64, 8)), ("elem", 4, 6, 357140, (4, 8, 64, 4)), ("elem", 8, 8, 138888, (4, 8, 64, 8))])
def test_fp32_few_nodes_many_operators(kernel, layout, N, F, E, want):
    """Up to N = 12 with more columns than the warp engine takes: register blocks, tile and unrolling."""
    v, _ = default(kernel, E, N, F, layout, "fp32")
    assert lc.variant_dict(v)["engine"] == "simt"
    assert (v.elems_per_thread, v.split_i, v.tile_e, v.unroll) == want


@pytest.mark.parametrize("layout", ["elem", "node"])
@pytest.mark.parametrize("N,F,E,engine", [(95, 8, 818, "simt"), (66, 8, 1178, "simt"), (84, 6, 1536, "simt"),
                                          (84, 6, 1537, "ksplit"), (84, 5, 900, "ksplit"), (64, 8, 1214, "ksplit"),
                                          (96, 8, 800, "ksplit")])
def test_fp32_few_elements_many_columns(kernel, layout, N, F, E, engine):
    """K-split CTAs walk their tile's column blocks: with few tiles of many columns the SIMT kernel, whose
    column blocks are CTAs, uses more of the GPU."""
    v, p = default(kernel, E, N, F, layout, "fp32")
    assert lc.variant_dict(v)["engine"] == engine
    if engine == "simt":
        assert p["column_blocks"] >= F


@pytest.mark.parametrize("layout", ["elem", "node"])
@pytest.mark.parametrize("N,F,chunk", [(176, 1, 16), (177, 3, 8), (185, 2, 8), (200, 3, 8), (201, 3, 16), (120, 3, 16)])
def test_ksplit_chunks_leave_room_for_two_ctas(kernel, layout, N, F, chunk):
    """Chunks of 8 where two CTAs of 128 elements then share an SM's 228 KB and with 16 they would not."""
    v, p = default(kernel, 400000, N, F, layout, "fp32")
    assert (v.tile_e, v.unroll) == (128, chunk)
    if N <= 200:
        assert 2 * (p["smem_bytes"] + 1024) <= 228 * 1024


@pytest.mark.parametrize("N,F,stages", [(27, 4, 2), (33, 3, 2), (35, 3, 2), (44, 2, 2), (47, 2, 2), (29, 3, 3), (20, 4, 3),
                                        (50, 1, 3)])
def test_bf16_element_major_stages(kernel, N, F, stages):
    """A third stage for narrow outputs only."""
    v, _ = default(kernel, 700000, N, F, "elem", "bf16")
    assert v.stages == stages


@pytest.mark.parametrize("N,F,want", [(65, 3, (2, 2)), (66, 3, (2, 2)), (79, 3, (2, 2)), (66, 2, (1, 3)), (84, 3, (1, 2))])
def test_bf16_node_major_three_operators(kernel, N, F, want):
    """Two threads a row and two stages for three operators between N = 65 and 79."""
    v, _ = default(kernel, 378784, N, F, "node", "bf16")
    assert (v.unroll, v.stages) == want


@pytest.mark.parametrize("E", [1, 5, 127, 130, 131])
def test_short_node_major_rows_keep_the_aligned_plan(kernel, E):
    """Rows off the 16-byte boundary with no 132nd value are never fetched in bulk: the wider stage rows
    for that must not cost an operator of the block or an A buffer."""
    for N, F in ((126, 3), (128, 4), (112, 4), (35, 3)):
        for precision in ("bf16", "bf16x3"):
            v, p = default(kernel, 128, N, F, "node", precision)
            q = lc.variant_plan(kernel, E, N, F, v)
            for key in ("ops_per_block", "a_buffers", "a_in_tmem", "smem_bytes"):
                assert q[key] == p[key], (N, F, precision, key)


@pytest.mark.parametrize("layout", ["elem", "node"])
@pytest.mark.parametrize("precision", ["fp32", "fp64", "bf16", "bf16x3"])
def test_default_is_among_the_candidates(kernel, layout, precision):
    """The exhaustive autotuner must not miss what a program gets without it."""
    for N, F in ((4, 1), (4, 6), (20, 2), (35, 3), (50, 1), (66, 3), (84, 4), (120, 3), (165, 3), (200, 1)):
        for E in (800, 20000, 1 << 21):
            v = lc.variant_dict(lc.variant_default(kernel, E, N, F, layout, precision))
            if lc.variant_plan(kernel, E, N, F, lc.Variant(**v))["threads"] >= 64:
                cands = [lc.variant_dict(c) for c in lc.enumerate_variants(kernel, E, N, F, layout, precision)]
                assert cands.count(v) == 1, (N, F, E)


@pytest.mark.parametrize("N,stages,copies", [(4, 1, False), (16, 1, False), (17, 1, True), (35, 1, True), (16, 2, True),
                                             (16, 3, True)])
def test_one_stage_of_short_unaligned_rows_is_read_directly(kernel, N, stages, copies):
    """Node-major rows off the 16-byte boundary: bulk copies take stage rows of 132 values, 16 bytes more (before
    the parts are aligned)."""
    v = lc.Variant(engine="tcgen05", layout="node", precision="bf16x3", tile_e=128, elems_per_thread=64, split_i=0,
                   unroll=3, prefetch_smem=1, stages=stages)
    aligned, odd = (lc.variant_plan(kernel, E, N, 2, v)["smem_bytes"] for E in (4000, 4001))
    assert (odd > aligned) if copies else (odd == aligned)
