"""Kernels whose CTAs walk several tiles, where other tests give every CTA one: the K-split kernel's
narrow column blocks (the D^T source wraps to block 0 of the next tile, the u buffer or buffers are
refilled) and early stage release.  Integer-valued inputs: bit-exact against the oracle."""

import numpy as np
import pytest

import oracle
import synth
from paper_1405_7470_gb300 import lc
from tests.test_parity_tc import run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kernel():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return lc.Kernel()


@pytest.mark.parametrize("layout", ["elem", "node"])
@pytest.mark.parametrize("N,F", [(73, 4), (75, 3), (84, 4), (64, 1), (65, 1), (113, 1), (165, 1)])
def test_ksplit_column_blocks(kernel, layout, N, F):
    E = 1501
    D, u = synth.integer_operands(E, N, F, seed=N)
    uu = synth.to_node_major(u) if layout == "node" else u
    want = oracle.contract(D, uu, layout)
    for tile_e in (64, 128):
        for chunk in (8, 16):
            for stages in (1, 2):
                v = lc.Variant(engine="ksplit", layout=layout, precision="fp32", tile_e=tile_e, elems_per_thread=8,
                               split_i=8, unroll=chunk, prefetch_smem=1, stages=stages, max_ctas=2)
                assert lc.variant_validate(kernel, E, N, F, v) == 0
                p = lc.variant_plan(kernel, E, N, F, v)
                assert p["grid"] == 2 and p["tiles"] >= 12
                assert np.array_equal(run(lc, kernel, v, D, uu, layout), want), (tile_e, chunk, stages)


@pytest.mark.parametrize("layout", ["elem", "node"])
@pytest.mark.parametrize("prec,N,F,combos", [
    ("bf16x3", 96, 2, [(1, 64, 2, 2), (1, 1, 1, 2), (1, 16, 2, 2)]),
    ("bf16x3", 48, 4, [(1, 64, 0, 2), (1, 1, 1, 3), (2, 16, 2, 2)]),
    ("bf16x3", 35, 3, [(1, 64, 1, 3), (2, 16, 1, 2)]),
    ("bf16", 64, 2, [(1, 64, 0, 2), (2, 32, 2, 2), (2, 16, 1, 3)])])
def test_early_release(kernel, layout, prec, N, F, combos):
    """Every descriptor is valid, and no conversion thread has more than the three chunks of 8 nodes that
    the early path takes (2 to 4 threads a row for unroll 2, else as many as epilogue threads, 3 at most)."""
    E = 20004
    D, u = synth.integer_operands(E, N, F, seed=N)
    uu = synth.to_node_major(u) if layout == "node" else u
    want = oracle.contract(D, uu, layout)
    for stages, kbw, aop, unroll in combos:
        v = lc.Variant(engine="tcgen05", layout=layout, precision=prec, tile_e=128, elems_per_thread=kbw, split_i=0,
                       unroll=unroll, prefetch_smem=2, stages=stages, store_rows=0 if layout == "node" else 32,
                       a_operand=aop, max_ctas=12)
        assert lc.variant_validate(kernel, E, N, F, v) == 0, (stages, kbw, aop)
        chunks = (N + 7) // 8
        threads = max(2, min(4, (chunks + 2) // 3)) if unroll == 2 else 3
        assert (chunks + threads - 1) // threads <= 3
        assert np.array_equal(run(lc, kernel, v, D, uu, layout), want), (stages, kbw, aop)
