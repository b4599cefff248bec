"""Which launch serves a group of a tensor-core grouped plan, and the grouped launch with CTAs that
walk many tiles of large groups (a launch of their own is switched off by max_ctas), against the CPU
FP64 oracle."""

import numpy as np
import pytest

import oracle
import synth
from tests.test_parity_grouped_tc import _check_sampled, make_groups, tc_variant

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lc():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1405_7470_gb300 import lc as lcmod
    lcmod.load()
    return lcmod


# two groups that would hold the GPU for more than 30 us beside tiny ones
SIZES = [(4, 700), (84, 1 << 18), (10, 33), (35, (1 << 18) + 77)]


@pytest.mark.parametrize("layout", ["elem", "node"])
def test_large_groups_stride_in_the_grouped_launch(lc, layout):
    kernel = lc.Kernel()
    data = synth.grouped_operands(SIZES, F=3, seed=2)
    v = tc_variant(lc, layout, "bf16x3")
    v.max_ctas = 20
    info = _check_sampled(lc, kernel, v, SIZES, data, layout)
    # one segment a CTA and no other launch: 4098 tiles and more on at most one CTA an SM
    assert info["segments"] == info["grid"] and 100 <= info["grid"] <= lc.device_info()["sm_count"]


def fields(lc, v):
    return {k: x for k, x in lc.variant_dict(v).items() if k != "layout"}


@pytest.mark.parametrize("layout", ["elem", "node"])
def test_large_groups_get_their_own_launch(lc, layout):
    import torch
    kernel = lc.Kernel()
    groups = []
    for N, E in SIZES:
        shape = (N, E) if layout == "node" else (E, N)
        groups.append((torch.ones((3, N, N), device="cuda"), torch.ones(shape, device="cuda"),
                       torch.empty((3,) + shape, device="cuda")))
    for kept in ({}, dict(max_ctas=20), dict(split_i=1), dict(a_operand=1), dict(mma_order=2)):
        v = tc_variant(lc, layout, "bf16x3")
        for name, x in kept.items():
            setattr(v, name, x)
        plan = lc.GroupedPlan(kernel, v, groups, use_graph=False)
        plan.run()
        torch.cuda.synchronize()
        assert lc.device_error() == 0
        for k, ((N, E), (_, _, out)) in enumerate(zip(SIZES, groups)):
            assert bool((out == N).all()), (N, kept)
            got = plan.group_variant(k)
            own = fields(lc, got) == fields(lc, lc.variant_default(kernel, E, N, 3, layout, "bf16x3"))
            assert own == (not kept and E > 100000), (N, kept)
            assert all(getattr(got, name) == x for name, x in kept.items()), (N, kept)
        del plan
