"""The K-split kernel's column blocks (64, 80, 96, 112 and 128 columns, chosen by the columns they
pad): sizes that take each of them, one column below and past a block's edge, and tiles of 64 and
128 elements.  Integer-valued inputs whose sums FP32 holds exactly: bit-exact against the oracle."""

import numpy as np
import pytest

import oracle
from paper_1405_7470_gb300 import lc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,F", [
    (64, 1), (65, 1), (80, 1), (81, 1), (96, 1), (97, 1), (112, 1), (113, 1), (128, 1), (129, 1),
    (73, 4), (75, 3), (84, 4), (165, 1)])
@pytest.mark.parametrize("layout", ["elem", "node"])
@pytest.mark.parametrize("tile_e", [64, 128])
def test_column_blocks_bit_exact(N, F, layout, tile_e):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    E = 389
    rng = np.random.default_rng(N * F)
    D = rng.integers(-8, 9, (F, N, N)).astype(np.float32)
    u = rng.integers(-8, 9, (E, N)).astype(np.float32)
    k = lc.Kernel()
    v = lc.Variant(engine="ksplit", layout=layout, precision="fp32", tile_e=tile_e, elems_per_thread=8, split_i=8,
                   unroll=16, prefetch_smem=1, stages=1)
    assert lc.variant_validate(k, E, N, F, v) == 0
    uu = u if layout == "elem" else u.T
    out = lc.contract(k, v, torch.from_numpy(D).cuda(), torch.from_numpy(np.ascontiguousarray(uu)).cuda())
    torch.cuda.synchronize()
    assert lc.device_error() == 0
    want = oracle.contract_rows(D, u, np.arange(E))
    got = out.cpu().numpy().astype(np.float64)
    if layout == "node":
        got = got.transpose(0, 2, 1)
    assert np.array_equal(got, np.asarray(want).reshape(got.shape))
