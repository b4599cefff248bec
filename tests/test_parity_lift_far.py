"""The surface lift's traces outside the window, gathered a row's half at a time over neighbouring
lanes: every length of a half, missing rows, indexes out of range in either half.  Integer-valued
inputs whose sums FP32 holds exactly: bit-exact against the oracle."""

import numpy as np
import pytest

import oracle
from paper_1405_7470_gb300 import lc

pytestmark = pytest.mark.gpu

# halves of 4, 8, 12, 16, 20, 24, 28 and 32 face nodes, with and without padding
SHAPES = [(10, 1, 3), (9, 2, 4), (13, 1, 13), (16, 4, 4), (20, 3, 7), (24, 2, 12), (27, 3, 9), (30, 1, 30), (33, 4, 10),
          (20, 3, 15), (36, 4, 12), (35, 4, 14), (40, 3, 19), (40, 4, 15), (24, 4, 16), (35, 4, 16)]


def problem(E, N, Nf, Nfp):
    rng = np.random.default_rng(E + 7 * N + Nfp)
    M = Nf * Nfp
    L = rng.integers(-3, 4, (N, M)).astype(np.float32)
    fmask = rng.integers(0, N, M).astype(np.int32)
    vmapP = rng.integers(0, E * N, (E, M)).astype(np.int32)
    # a third of the faces keeps its neighbour in the window, so that rows mix both kinds
    near = (np.arange(E)[:, None] * N + rng.integers(0, N, (E, M))).astype(np.int32)
    vmapP = np.where(np.repeat(rng.random((E, Nf)) < 0.33, Nfp, axis=1), near, vmapP)
    s = rng.integers(1, 4, (E, Nf)).astype(np.float32)
    u = rng.integers(-8, 9, (E, N)).astype(np.float32)
    return L, fmask, vmapP, s, u


def dev(*arrays):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in arrays]


@pytest.mark.parametrize("N,Nf,Nfp", SHAPES)
def test_bit_exact(N, Nf, Nfp):
    k = lc.Kernel(lc.LIFT_DOMAIN, lc.LIFT_INSTRUCTION)
    for E, ctas in ((1, 0), (31, 0), (97, 0), (2500, 1), (20011, 0), (20011, 3)):
        args = problem(E, N, Nf, Nfp)
        v = lc.variant_default(k, E, N, 1, "elem", "fp32")
        v.max_ctas = ctas
        out = lc.lift(k, v, *dev(*args))
        assert lc.device_error() == 0
        assert np.array_equal(out.cpu().numpy().astype(np.float64), oracle.lift(*args)), (E, ctas)


@pytest.mark.parametrize("N,Nf,Nfp", SHAPES[1::3])
def test_out_of_range(N, Nf, Nfp):
    """Indexes out of range in the first and the second half of rows: NaN in those rows alone."""
    k = lc.Kernel(lc.LIFT_DOMAIN, lc.LIFT_INSTRUCTION)
    E, M = 3001, Nf * Nfp
    L, fmask, vmapP, s, u = problem(E, N, Nf, Nfp)
    L[:] = np.where(L == 0, 1, L)  # every flux reaches every output
    want = oracle.lift(L, fmask, vmapP, s, u)
    bad = {3: 0, 40: M - 1, 77: M // 2, E - 1: M - 1}
    for value in (E * N, -1, 2 ** 31 - 1):
        broken = vmapP.copy()
        for e, m in bad.items():
            broken[e, m] = value
        v = lc.variant_default(k, E, N, 1, "elem", "fp32")
        out = lc.lift(k, v, *dev(L, fmask, broken, s, u))
        assert lc.device_error() == 11  # LC_ERR_INDEX (and cleared)
        got = out.cpu().numpy().astype(np.float64)
        rows = sorted(bad)
        assert np.all(np.isnan(got[rows]))
        assert np.array_equal(np.delete(got, rows, axis=0), np.delete(want, rows, axis=0))
