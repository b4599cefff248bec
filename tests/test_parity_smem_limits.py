"""A kernel instance serves plans of different shared-memory sizes in any order: a grouped plan
without a graph still runs after smaller launches and plans on the same instances, and its groups
may come largest first.  Results against the CPU FP64 oracle."""

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


def fp32_variant(lc, layout):
    return lc.Variant(layout=layout, elems_per_thread=4, split_i=8, unroll=4, prefetch_smem=1, stages=2, ctas_per_sm=2)


def tc_variant(lc, layout):
    return lc.Variant(engine="tcgen05", layout=layout, precision="bf16x3", tile_e=128, elems_per_thread=64, split_i=0,
                      unroll=3, prefetch_smem=1, stages=1, store_rows=0 if layout == "node" else 128)


def make(sizes, layout, seed=3):
    import torch
    groups, host = [], []
    for (N, E), (D, u) in zip(sizes, synth.grouped_operands(sizes, F=3, seed=seed)):
        uu = synth.to_node_major(u) if layout == "node" else u
        groups.append((to_dev(D), to_dev(uu), torch.empty((3, N, E) if layout == "node" else (3, E, N), device="cuda")))
        host.append((D, uu))
    return groups, host


def check(lc, plan, groups, host, layout):
    """Run and compare within the FP32 FMA bound (three-term sums: six products a term, doubled)."""
    import torch
    for _, _, out in groups:
        out.fill_(float("nan"))
    plan.run()
    torch.cuda.synchronize()
    assert lc.device_error() == 0
    for k, ((D, u), (_, _, out)) in enumerate(zip(host, groups)):
        factor = 1 if lc.variant_dict(plan.group_variant(k))["precision"] == "fp32" else 16
        ref = oracle.contract(D, u, layout)
        err = np.abs(out.cpu().numpy().astype(np.float64) - ref)
        assert np.all(err <= factor * fma_bound(D, u, layout, 2.0 ** -24)), (D.shape, layout)


@pytest.mark.parametrize("layout", ["elem", "node"])
def test_contraction_between_runs(lc, layout):
    import torch
    kernel = lc.Kernel()
    sizes = [(165, 300)]
    groups, host = make(sizes, layout)
    plan = lc.GroupedPlan(kernel, fp32_variant(lc, layout), groups, use_graph=False)
    assert lc.variant_dict(plan.group_variant(0))["engine"] == "ksplit"
    check(lc, plan, groups, host, layout)
    ks = plan.group_variant(0)
    threads = lc.variant_plan(kernel, 300, 165, 3, ks)["threads"]
    shared = 0
    for N in (64, 75, 84, 100, 120, 128):  # the same instance where the column block is as wide
        shared += lc.variant_plan(kernel, 200, N, 3, ks)["threads"] == threads
        D, u = torch.ones((3, N, N), device="cuda"), torch.ones((N, 200) if layout == "node" else (200, N), device="cuda")
        assert torch.all(lc.contract(kernel, ks, D, u) == N)
    assert shared
    check(lc, plan, groups, host, layout)


@pytest.mark.parametrize("graph", [True, False])
@pytest.mark.parametrize("layout", ["elem", "node"])
def test_largest_group_first(lc, layout, graph):
    import torch
    kernel = lc.Kernel()
    sizes = [(165, 300), (160, 129), (128, 200), (100, 150), (96, 260)]
    groups, host = make(sizes, layout)
    plan = lc.GroupedPlan(kernel, fp32_variant(lc, layout), groups, use_graph=graph, stream=torch.cuda.Stream())
    check(lc, plan, groups, host, layout)


@pytest.mark.parametrize("layout", ["elem", "node"])
@pytest.mark.parametrize("variant", [fp32_variant, tc_variant])
def test_smaller_plan_created_between(lc, variant, layout):
    kernel = lc.Kernel()
    groups, host = make([(84, 200), (20, 300)], layout)
    small, small_host = make([(4, 50)], layout)
    plan = lc.GroupedPlan(kernel, variant(lc, layout), groups, use_graph=False)
    other = lc.GroupedPlan(kernel, variant(lc, layout), small, use_graph=False)
    check(lc, plan, groups, host, layout)
    check(lc, other, small, small_host, layout)
    check(lc, plan, groups, host, layout)
