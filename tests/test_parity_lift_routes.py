"""Which kernel serves a surface lift: the tiled one (also asked for by two staging buffers, tiles of
128 or no prefetch, whose index check is tested here) where the one with the flux rows in registers
measured slower: rows of u that meet in one bank, long rows, and wide operators on few elements."""

import numpy as np
import pytest

import oracle
import synth
from paper_1405_7470_gb300 import lc

pytestmark = pytest.mark.gpu


def dev(*arrays):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in arrays]


@pytest.mark.parametrize("E,N,Nf,Nfp,accumulate,tiled", [
    (20000, 64, 4, 16, False, True), (20000, 32, 4, 10, False, True), (4099, 128, 4, 10, False, True),
    (30000, 50, 1, 30, False, True), (30000, 48, 3, 9, False, True), (4099, 27, 3, 9, False, True),
    (20000, 35, 4, 15, False, False), (4099, 35, 4, 15, False, False), (20000, 20, 4, 10, False, False),
    (4099, 20, 4, 10, False, False), (12000, 60, 4, 15, False, False), (20000, 64, 4, 16, True, True),
    (4099, 27, 3, 9, True, False), (12000, 50, 1, 30, True, False), (12000, 32, 4, 15, True, False),
    (12000, 64, 4, 15, True, True), (20000, 32, 4, 15, True, True)])
def test_kernel_by_shape(E, N, Nf, Nfp, accumulate, tiled):
    """Both kernels' sums differ in their last bits (the tiled kernel adds m in order, the other one the
    halves of m apart), so the bits tell which one ran."""
    rng = np.random.default_rng(N)
    M = Nf * Nfp
    L = rng.uniform(-1, 1, (N, M)).astype(np.float32)
    fmask = rng.integers(0, N, M).astype(np.int32)
    vmapP = rng.integers(0, E * N, (E, M)).astype(np.int32)
    s = rng.uniform(0.5, 2, (E, Nf)).astype(np.float32)
    u = rng.standard_normal((E, N)).astype(np.float32)
    k = lc.Kernel(lc.LIFT_DOMAIN, lc.LIFT_INSTRUCTION)
    d = dev(L, fmask, vmapP, s, u)
    got = lc.lift(k, lc.variant_default(k, E, N, 1, "elem", "fp32"), *d, accumulate=accumulate)
    v = lc.variant_default(k, E, N, 1, "elem", "fp32")
    v.stages = 2
    ref = lc.lift(k, v, *d, accumulate=accumulate)
    assert lc.device_error() == 0
    assert bool((got == ref).all()) == tiled


@pytest.mark.parametrize("fields", [dict(stages=2), dict(tile_e=128), dict(prefetch_smem=0)])
def test_tiled_kernel_reports_indexes(fields):
    k = lc.Kernel(lc.LIFT_DOMAIN, lc.LIFT_INSTRUCTION)
    L, fmask, vmapP, s, u = synth.surface_mesh(500, order=2, width=8, seed=2)
    want = oracle.lift(L, fmask, vmapP, s, u)
    for value in (u.size, u.size + 1000, -1):
        bad = vmapP.copy()
        bad[7, 3] = bad[499, 20] = value
        v = lc.variant_default(k, u.shape[0], u.shape[1], 1, "elem", "fp32")
        for name, x in fields.items():
            setattr(v, name, x)
        out = lc.lift(k, v, *dev(L, fmask, bad, s, u))
        assert lc.device_error() == 11  # LC_ERR_INDEX (and cleared)
        got = out.cpu().numpy()
        assert np.all(np.isnan(got[[7, 499]])) and np.all(np.isfinite(np.delete(got, [7, 499], axis=0)))
        assert oracle.rel_fro_error(np.delete(got, [7, 499], axis=0).astype(np.float64),
                                    np.delete(want, [7, 499], axis=0)) <= 1e-6
