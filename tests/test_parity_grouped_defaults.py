"""Grouped FP32 plans take the descriptors lc_variant_default gives from N = 13 on (whole rows in
registers, tiles, K-split): every group within the FP32 FMA bound of the CPU FP64 oracle."""

import numpy as np
import pytest

import oracle
import synth
from tests.gpu_util import fma_bound, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lc():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1405_7470_gb300 import lc as lcmod
    lcmod.load()
    return lcmod


SETS = [[(13, 300), (24, 129)], [(4, 700), (35, 513), (40, 257)], [(20, 200), (56, 130), (84, 300)],
        [(64, 131), (95, 260), (120, 150)], [(20, 1), (35, 0), (165, 140)]]


@pytest.mark.parametrize("layout", ["elem", "node"])
@pytest.mark.parametrize("sizes", SETS)
def test_default_descriptors(lc, sizes, layout):
    import torch
    kernel = lc.Kernel()
    groups, host = [], []
    for (N, E), (D, u) in zip(sizes, synth.grouped_operands(sizes, F=3, seed=9)):
        uu = synth.to_node_major(u) if layout == "node" else u
        groups.append((to_dev(D), to_dev(uu), torch.empty((3, N, E) if layout == "node" else (3, E, N), device="cuda")))
        host.append((D, uu))
    for N, E in sizes:
        if N < 13 or E == 0:
            continue
        v = lc.variant_default(kernel, E, N, 3, layout, "fp32")
        for graph in (True, False):
            plan = lc.GroupedPlan(kernel, v, groups, use_graph=graph, stream=torch.cuda.Stream())
            for _, _, out in groups:
                out.fill_(float("nan"))
            torch.cuda.synchronize()
            plan.run()
            torch.cuda.synchronize()
            assert lc.device_error() == 0
            for (D, u), (_, _, out) in zip(host, groups):
                err = np.abs(out.cpu().numpy().astype(np.float64) - oracle.contract(D, u, layout))
                assert np.all(err <= fma_bound(D, u, layout, 2.0 ** -24)), (D.shape, N, layout)
            engine = lc.variant_dict(v)["engine"]
            for k, (n, e) in enumerate(sizes):
                if e > 0:
                    ks = n >= (64 if engine == "ksplit" else 96)
                    assert lc.variant_dict(plan.group_variant(k))["engine"] == ("ksplit" if ks else "simt"), (n, N)


@pytest.mark.parametrize("layout", ["elem", "node"])
def test_refused_as_before(lc, layout):
    """The warp engine, FP64, guard-free tails, unroll 2, 8 without a staged u, and K-split descriptors
    that no plain call takes are refused."""
    import torch
    kernel = lc.Kernel(assumptions="E mod 128 = 0")
    D, u = torch.ones((3, 35, 35), device="cuda"), torch.ones((35, 128) if layout == "node" else (128, 35), device="cuda")
    groups = [(D, u, torch.empty((3, 35, 128) if layout == "node" else (3, 128, 35), device="cuda"))]
    ks = dict(engine="ksplit", tile_e=128, elems_per_thread=8, split_i=8, unroll=16)
    for bad in (dict(engine="warp", elems_per_thread=1, split_i=1, unroll=1, prefetch_smem=0), dict(precision="fp64"),
                dict(tail_free=1), dict(unroll=2), dict(unroll=8, prefetch_smem=0), dict(unroll=8, tail_free=1),
                dict(ks, tail_free=1), dict(ks, tile_e=96), dict(ks, unroll=4), dict(ks, stages=3)):
        with pytest.raises(lc.LcError):
            lc.GroupedPlan(kernel, lc.Variant(layout=layout, **bad), groups, use_graph=False)
