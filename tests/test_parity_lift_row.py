"""The surface lift with the flux rows in registers (lift_row.cu: up to four faces, up to 64 face
nodes) at the edges of its tiles: halves of the face nodes with and without padding, rows whose
index list is no multiple of 16 bytes, chunks with missing rows, one CTA for every tile, traces
anywhere in u (most of them outside the window), out off the 16-byte boundary; and the shapes just
beyond it.  Integer-valued inputs whose sums FP32 holds exactly: bit-exact against the oracle."""

import numpy as np
import pytest

import oracle
from paper_1405_7470_gb300 import lc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("accumulate", [False, True])
@pytest.mark.parametrize("E,N,Nf,Nfp", [
    (1, 1, 1, 1), (33, 3, 1, 5), (97, 10, 3, 7), (65, 35, 4, 15), (4099, 35, 4, 15), (3001, 20, 2, 9),
    (40000, 13, 3, 8), (700, 64, 4, 16), (515, 9, 1, 33), (1000, 100, 2, 4), (300, 128, 4, 16),
    (1000, 7, 5, 4), (1000, 12, 3, 22)])
def test_shapes_bit_exact(accumulate, E, N, Nf, Nfp):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(E + N)
    M = Nf * Nfp
    L = rng.integers(-3, 4, (N, M)).astype(np.float32)
    fmask = rng.integers(0, N, M).astype(np.int32)
    vmapP = rng.integers(0, E * N, (E, M)).astype(np.int32)
    near = (np.arange(E)[:, None] * N + rng.integers(0, N, (E, M))).astype(np.int32)
    vmapP = np.where(rng.random((E, 1)) < 0.5, near, vmapP)  # half of the elements inside the window
    s = rng.integers(1, 4, (E, Nf)).astype(np.float32)
    u = rng.integers(-8, 9, (E, N)).astype(np.float32)
    out0 = rng.integers(-5, 6, (E, N)).astype(np.float32)
    want = oracle.lift(L, fmask, vmapP, s, u, out=out0 if accumulate else None)
    k = lc.Kernel(lc.LIFT_DOMAIN, lc.LIFT_INSTRUCTION)
    Ld, fd, vd, sd, ud = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (L, fmask, vmapP, s, u))
    for ctas, shift in ((0, 0), (1, 0), (2, 1)):
        v = lc.variant_default(k, E, N, 1, "elem", "fp32")
        v.max_ctas = ctas
        out = torch.empty(E * N + 4, device="cuda")[shift:shift + E * N].view(E, N)
        out.copy_(torch.from_numpy(out0))
        lc.lift(k, v, Ld, fd, vd, sd, ud, out, accumulate=accumulate)
        torch.cuda.synchronize()
        assert lc.device_error() == 0
        assert np.array_equal(out.cpu().numpy().astype(np.float64), want), (ctas, shift)
