"""GPU parity of the three-term plans with the A terms in tensor memory and the products stacked
(regions 8-column aligned), and of early stage release where the stage reads queue behind bank
conflicts, against the CPU FP64 oracle.

Bars: integer-valued inputs bit-exact; random inputs within twice the FP32-accumulation bound of
the exact contraction of the split operands.
"""

import numpy as np
import pytest

import oracle
import synth
from tests.test_parity_tc import accum_bound, run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lc():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1405_7470_gb300 import lc as lcmod
    lcmod.load()
    return lcmod


def descriptor(lc, layout, split, unroll, prefetch, stages, kbw, rows):
    return lc.Variant(engine="tcgen05", layout=layout, precision="bf16x3", tile_e=128, elems_per_thread=kbw,
                      split_i=split, unroll=unroll, prefetch_smem=prefetch, stages=stages,
                      store_rows=0 if layout == "node" else rows, a_operand=2)


# (E, N, operators per block, F): one operator at the largest N that stacks (88) and below it, CB a
# multiple of 8 but not of 16 (N = 84, 20, 36), several operators per block, one tile and several
@pytest.mark.parametrize("layout", ["elem", "node"])
@pytest.mark.parametrize("E,N,split,F", [(20111, 88, 1, 2), (20112, 84, 1, 4), (127, 70, 1, 1), (129, 56, 1, 3),
                                         (30000, 20, 3, 3), (4099, 36, 2, 2), (1, 9, 1, 1)])
def test_stacked_in_tensor_memory(lc, layout, E, N, split, F):
    kernel = lc.Kernel()
    Di, ui = synth.integer_operands(E, N, F, seed=E + N)
    D, u = synth.operands(E, N, F, np.float32, seed=N, scale_exp=3.0)
    tr = synth.to_node_major if layout == "node" else np.asarray
    want = oracle.contract(Di, tr(ui), layout)
    target = oracle.contract_bf16x3(D, tr(u), layout)
    Ds, us = oracle.bf16_split3(D), oracle.bf16_split3(tr(u))
    bound = accum_bound(sum(np.abs(x) for x in Ds), sum(np.abs(x) for x in us), layout, "bf16x3")
    for unroll, prefetch, stages, kbw, rows in ((2, 1, 2, 64, 32), (3, 2, 1, 1, 128), (1, 2, 1, 32, 32)):
        v = descriptor(lc, layout, split, unroll, prefetch, stages, kbw, rows)
        assert lc.variant_validate(kernel, E, N, F, v) == 0
        p = lc.variant_plan(kernel, E, N, F, v)
        assert p["a_in_tmem"] == 1 and p["stacked"] == 1
        assert np.array_equal(run(lc, kernel, v, Di, tr(ui), layout), want), (unroll, kbw)
        assert np.all(np.abs(run(lc, kernel, v, D, tr(u), layout) - target) <= bound), (unroll, kbw)


# element-major rows of 48 and 96 values: the 16-byte reads of a warp hit the same banks 4 and 8 times
@pytest.mark.parametrize("prec,N,F", [("bf16x3", 96, 2), ("bf16x3", 48, 4), ("bf16", 64, 2)])
def test_early_release_with_queued_stage_reads(lc, prec, N, F):
    kernel = lc.Kernel()
    E = 100000
    D, u = synth.integer_operands(E, N, F, seed=N)
    want = oracle.contract(D, u)
    for stages, kbw, aop in ((1, 64, 0), (2, 1, 2), (1, 64, 2)):
        v = lc.Variant(engine="tcgen05", layout="elem", precision=prec, tile_e=128, elems_per_thread=kbw, split_i=0,
                       unroll=2, prefetch_smem=2, stages=stages, store_rows=32, a_operand=aop)
        if lc.variant_validate(kernel, E, N, F, v) != 0:
            continue
        assert np.array_equal(run(lc, kernel, v, D, u, "elem"), want), (stages, kbw, aop)


# node-major rows that start off the 16-byte boundary by each amount, tiles before and at the
# point where the last tile's copies would run past the array, N off every chunk size
@pytest.mark.parametrize("prec", ["bf16", "bf16x3"])
@pytest.mark.parametrize("E", [128 * 3 + 1, 128 * 3 + 2, 128 * 3 + 3, 128 * 3 + 5, 128 * 3 + 7, 30001, 30002, 131, 130])
def test_node_major_unaligned_rows(lc, prec, E):
    kernel = lc.Kernel()
    for N, F in ((20, 2), (35, 3), (9, 1)):
        D, u = synth.integer_operands(E, N, F, seed=E + N)
        uu = synth.to_node_major(u)
        want = oracle.contract(D, uu, "node")
        for unroll, prefetch, stages in ((1, 1, 3), (3, 2, 1)):
            v = lc.Variant(engine="tcgen05", layout="node", precision=prec, tile_e=128, elems_per_thread=64, split_i=0,
                           unroll=unroll, prefetch_smem=prefetch, stages=stages, store_rows=0, max_ctas=40)
            assert lc.variant_validate(kernel, E, N, F, v) == 0
            assert np.array_equal(run(lc, kernel, v, D, uu, "node"), want), (N, unroll)
