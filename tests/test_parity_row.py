"""GPU parity of the FP32 row kernel (SIMT engine, j wholly unrolled: unroll 8 with the u tile
staged, N = 13 to 40) against the CPU FP64 oracle: integer-valued inputs bit-exact, random inputs
within the FP32 FMA-chain bound, sentinels around every output untouched."""

import numpy as np
import pytest

import oracle
import synth
from tests.gpu_util import CanaryOut, fma_bound, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lc():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1405_7470_gb300 import lc as lcmod
    lcmod.load()
    return lcmod


def run(lc, v, D, u, layout):
    import torch
    F, N, _ = D.shape
    E = u.shape[1] if layout == "node" else u.shape[0]
    co = CanaryOut((F, N, E) if layout == "node" else (F, E, N), np.float32)
    lc.contract(lc.Kernel(), v, to_dev(D), to_dev(u), co.out)
    torch.cuda.synchronize()
    assert lc.device_error() == 0
    assert co.intact(), "write outside the output"
    return co.out.cpu().numpy().astype(np.float64)


# the ends of the range of N, each residue mod 4; one element, chunk edges, unaligned outputs
# (E N % 4 != 0), batches of one operator a unit, of whole chunks (2 and 4 rows a thread), and
# several chunks a warp (max_ctas)
@pytest.mark.parametrize("layout", ["elem", "node"])
@pytest.mark.parametrize("E,N,F,max_ctas", [(1, 13, 1, 0), (63, 16, 2, 0), (65, 17, 3, 0), (4099, 35, 3, 0), (129, 40, 8, 0),
                                            (20000, 14, 4, 3), (20002, 35, 2, 3), (40001, 39, 3, 5), (160001, 21, 1, 0),
                                            (160000, 40, 2, 20), (156000, 22, 2, 7)])
def test_row_kernel(lc, layout, E, N, F, max_ctas):
    kernel = lc.Kernel()
    v = lc.Variant(layout=layout, tile_e=64, elems_per_thread=4, split_i=8, unroll=8, prefetch_smem=1, stages=2,
                   ctas_per_sm=2, max_ctas=max_ctas)
    assert lc.variant_validate(kernel, E, N, F, v) == 0
    tr = synth.to_node_major if layout == "node" else np.asarray
    D, u = synth.integer_operands(E, N, F, seed=E + N)
    assert np.array_equal(run(lc, v, D, tr(u), layout), oracle.contract(D, tr(u), layout))
    D, u = synth.operands(E, N, F, np.float32, seed=N, scale_exp=3.0)
    got = run(lc, v, D, tr(u), layout)
    ref = oracle.contract(D, tr(u), layout)
    assert np.all(np.abs(got - ref) <= fma_bound(D, tr(u), layout, 2.0 ** -24))
