"""The work that is timed: calls of the library's public entry points at the sizes they are used at.

Every case names an entry point (``op``), its sizes, layout and precision.  Inputs are drawn
on the GPU from a seed: operators uniform on [-1, 1), fields standard normal, as the
synthetic workloads of this repository draw them.  The descriptor of a contraction is the
library's default for the problem, as a program that does not tune would take it.
"""

from __future__ import annotations

import math

import torch

from paper_1405_7470_gb300 import lc

GROUP_NS = (4, 10, 20, 35, 56, 84, 120, 165)
# floor(2^U(14, 21)) from seed 0: the uneven-batching workload's element counts
GROUP_ES = (360273, 60662, 19987, 17751, 847522, 1373370, 310977, 564445)


def _contract(name, E, N, F, layout, precision, scale=False):
    return dict(name=name, op="contract", E=E, N=N, F=F, layout=layout, precision=precision, scale=scale)


def listed():
    groups = dict(op="grouped", F=3, layout="elem", precision="bf16x3", groups=len(GROUP_NS))
    for g, (n, e) in enumerate(zip(GROUP_NS, GROUP_ES)):
        groups[f"N{g}"], groups[f"E{g}"] = n, e
    return [
        # one operator on one small mesh partition in double precision: a call whose launch and
        # latency count, the smallest of the set
        _contract("fp64_elem_n20_f1_e4096", 4096, 20, 1, "elem", "fp64"),
        # the three reference derivatives of degree-4 tetrahedra over a large mesh, FP32 FMA
        _contract("fp32_elem_n35_f3_e2m", 1 << 21, 35, 3, "elem", "fp32"),
        # the same work at FP32-level accuracy on the tensor cores, in both layouts a solver keeps
        _contract("bf16x3_elem_n35_f3_e2m", 1 << 21, 35, 3, "elem", "bf16x3"),
        _contract("bf16x3_node_n35_f3_e2m", 1 << 21, 35, 3, "node", "bf16x3"),
        # a mesh partition of odd size, degree 3, two derivatives: a few waves of tiles, no
        # 16-byte rows
        _contract("bf16x3_node_n20_f2_e19987", 19987, 20, 2, "node", "bf16x3"),
        # degree-6 elements, four operators, fields of very different scales per element
        _contract("bf16x3_elem_n84_f4_e1m", 1 << 20, 84, 4, "elem", "bf16x3", scale=True),
        _contract("bf16_elem_n84_f4_e1m", 1 << 20, 84, 4, "elem", "bf16", scale=True),
        # degree-7 elements, odd element count, node-major: rows of u and out start unaligned
        _contract("fp32_node_n120_f3_e310977", 310977, 120, 3, "node", "fp32"),
        # eight groups of mixed degree in one plan, replayed from its graph (the largest)
        dict(groups, name="grouped_bf16x3_8_groups"),
        # physical derivatives: the three reference derivatives mixed by each element's factors
        dict(name="geo_bf16x3_elem_n35_f3_e2m", op="geo", E=1 << 21, N=35, F=3, layout="elem", precision="bf16x3"),
        # the surface term of a degree-4 tetrahedral mesh numbered for locality
        dict(name="lift_n35_e2m", op="lift", E=1 << 21, degree=4, width=64, accumulate=0),
        # the streaming update of a time step
        dict(name="saxpy_2p28", op="saxpy", n=1 << 28),
    ]


def _log_uniform(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))


def draw(rng):
    """A case of the same ranges: N 4 to 165, E 2^12 to 2^22, F 1 to 4 and every path; sizes whose
    cost would pass the largest listed case's are cut in E."""
    kind = rng.random()
    if kind < 0.62:
        precision = rng.choice(("fp32", "fp32", "bf16", "bf16x3", "bf16x3", "fp64"))
        layout = rng.choice(("elem", "node"))
        if precision == "fp64":
            N, F = rng.randint(4, 32), 1
            E = _log_uniform(rng, 1 << 12, 1 << 18)
        else:
            N, F = rng.randint(4, 165), rng.randint(1, 4)
            E = _log_uniform(rng, 1 << 12, 1 << 22)
            E = min(E, int(3.0e9 / (4 * N * (1 + F))), int(6.0e10 / (2 * N * N * F)))
        return dict(op="contract", E=E, N=N, F=F, layout=layout, precision=precision, scale=rng.random() < 0.25)
    if kind < 0.70:
        count = rng.randint(4, 8)
        c = dict(op="grouped", F=rng.randint(1, 3), layout=rng.choice(("elem", "node")),
                 precision=rng.choice(("fp32", "bf16x3", "bf16x3")), groups=count)
        for g, n in enumerate(sorted(rng.sample(GROUP_NS, count))):
            c[f"N{g}"] = n
            c[f"E{g}"] = min(_log_uniform(rng, 1 << 12, 1 << 19), int(6.0e9 / (n * n)))
        return c
    if kind < 0.80:
        F = rng.choice((2, 3))
        return dict(op="geo", E=_log_uniform(rng, 1 << 12, 1 << 21), N=rng.randint(4, 48 if F == 3 else 64), F=F,
                    layout=rng.choice(("elem", "node")), precision=rng.choice(("bf16", "bf16x3")))
    if kind < 0.92:
        degree = rng.randint(1, 6)
        nodes = (degree + 1) * (degree + 2) * (degree + 3) // 6
        return dict(op="lift", E=min(_log_uniform(rng, 1 << 12, 1 << 21), int(8.0e7 / nodes)), degree=degree,
                    width=rng.choice((16, 64, 200)), accumulate=rng.randint(0, 1))
    return dict(op="saxpy", n=_log_uniform(rng, 1 << 14, 1 << 28))


# ------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _dtype(precision):
    return torch.float64 if precision == "fp64" else torch.float32


def _operands(gen, E, N, F, layout, precision, scale=False):
    """(D, u): D uniform on [-1, 1), u standard normal, each element's row times 10^k, k uniform on
    [-3, 3), where fields of very different scales meet."""
    dt = _dtype(precision)
    D = torch.rand((F, N, N), generator=gen, dtype=dt, device="cuda").mul_(2).sub_(1)
    u = torch.randn((E, N), generator=gen, dtype=dt, device="cuda")
    if scale:
        k = torch.rand((E, 1), generator=gen, dtype=dt, device="cuda").mul_(6).sub_(3)
        u.mul_(torch.pow(10.0, k))
    return D, (u.t().contiguous() if layout == "node" else u)


def _out(E, N, F, layout, precision):
    return torch.empty((F, N, E) if layout == "node" else (F, E, N), dtype=_dtype(precision), device="cuda")


def _tet(degree):
    """Node count of a degree-`degree` tetrahedron and its four faces' node lists."""
    nodes = [(a, b, c) for a in range(degree + 1) for b in range(degree + 1 - a) for c in range(degree + 1 - a - b)]
    faces = [[k for k, p in enumerate(nodes) if on(*p)]
             for on in (lambda a, b, c: c == 0, lambda a, b, c: b == 0, lambda a, b, c: a == 0,
                        lambda a, b, c: a + b + c == degree)]
    return len(nodes), faces


def _mesh(E, degree, width):
    """(N, Nfp, fmask, vmapP) of a strip of tetrahedra: face 0 of element e meets face 1 of e + 1
    with its nodes reversed, face 2 meets face 3 of e + width; outer faces meet themselves."""
    N, faces = _tet(degree)
    Nfp = len(faces[0])
    fm = torch.tensor(faces, dtype=torch.int64, device="cuda")
    e = torch.arange(E, device="cuda")[:, None]
    vmapP = torch.empty((E, 4 * Nfp), dtype=torch.int32, device="cuda")
    for f, (off, fn, rev) in enumerate(((1, 1, True), (-1, 0, True), (width, 3, False), (-width, 2, False))):
        nb = e + off
        other = fm[fn].flip(0) if rev else fm[fn]
        inside = (nb >= 0) & (nb < E)
        vmapP[:, f * Nfp:(f + 1) * Nfp] = torch.where(inside, nb * N + other, e * N + fm[f]).int()
    return N, Nfp, fm.reshape(-1).int(), vmapP


def prepare(case, seed):
    """What a program holds before the call: inputs, output buffer, kernel handle, descriptor or plan."""
    gen = _gen(seed)
    op = case["op"]
    if op == "contract":
        E, N, F, layout, precision = (case[k] for k in ("E", "N", "F", "layout", "precision"))
        kernel = lc.Kernel()
        D, u = _operands(gen, E, N, F, layout, precision, case["scale"])
        return dict(op=op, kernel=kernel, v=lc.variant_default(kernel, E, N, F, layout, precision), D=D, u=u,
                    out=_out(E, N, F, layout, precision))
    if op == "grouped":
        F, layout, precision = case["F"], case["layout"], case["precision"]
        kernel = lc.Kernel()
        groups = []
        for g in range(case["groups"]):
            E, N = case[f"E{g}"], case[f"N{g}"]
            D, u = _operands(gen, E, N, F, layout, precision)
            groups.append((D, u, _out(E, N, F, layout, precision)))
        if precision == "fp32":
            v = lc.Variant(layout=layout, elems_per_thread=4, split_i=8, unroll=4, prefetch_smem=1, stages=2,
                           ctas_per_sm=2)
        else:
            v = lc.Variant(engine="tcgen05", layout=layout, precision=precision, tile_e=128, elems_per_thread=64,
                           split_i=0, unroll=3, prefetch_smem=1, stages=1, store_rows=0 if layout == "node" else 128)
        torch.cuda.synchronize()
        plan = lc.GroupedPlan(kernel, v, groups, use_graph=True, stream=torch.cuda.Stream())
        return dict(op=op, plan=plan, outs=[g[2] for g in groups])
    if op == "geo":
        E, N, F, layout, precision = (case[k] for k in ("E", "N", "F", "layout", "precision"))
        kernel = lc.Kernel(lc.GEO_DOMAIN, lc.GEO_INSTRUCTION)
        D, u = _operands(gen, E, N, F, layout, precision)
        r = torch.randn((F, F, E) if layout == "node" else (E, F, F), generator=gen, device="cuda")
        return dict(op=op, kernel=kernel, v=lc.variant_default(kernel, E, N, F, layout, precision), D=D, u=u, r=r,
                    out=_out(E, N, F, layout, precision))
    if op == "lift":
        E = case["E"]
        N, Nfp, fmask, vmapP = _mesh(E, case["degree"], case["width"])
        L = torch.rand((N, 4 * Nfp), generator=gen, device="cuda").mul_(2).sub_(1)
        s = torch.rand((E, 4), generator=gen, device="cuda").mul_(1.5).add_(0.5)
        u = torch.randn((E, N), generator=gen, device="cuda")
        kernel = lc.Kernel(lc.LIFT_DOMAIN, lc.LIFT_INSTRUCTION)
        return dict(op=op, kernel=kernel, v=lc.variant_default(kernel, E, N, 1, "elem", "fp32"), L=L, fmask=fmask,
                    vmapP=vmapP, s=s, u=u, out=torch.zeros((E, N), device="cuda"), accumulate=bool(case["accumulate"]))
    n = case["n"]
    kernel = lc.Kernel("{ [i]: 0<=i<n }", "z[i] = a*x[i] + y[i]")
    x = torch.randn(n, generator=gen, device="cuda")
    y = torch.randn(n, generator=gen, device="cuda")
    return dict(op="saxpy", kernel=kernel, v=lc.variant_default(kernel, n, 1, 1, "elem", "fp32"),
                arrays=[torch.empty(n, device="cuda"), x, y])


def run(state):
    """One call; the output is the state's own buffer."""
    op = state["op"]
    if op == "contract":
        return lc.contract(state["kernel"], state["v"], state["D"], state["u"], state["out"])
    if op == "grouped":
        state["plan"].run()
        return list(state["outs"])
    if op == "geo":
        return lc.contract_geo(state["kernel"], state["v"], state["D"], state["u"], state["r"], state["out"])
    if op == "lift":
        if state["accumulate"]:
            state["out"].zero_()  # the right-hand side starts from zero, the surface term adds to it
        return lc.lift(state["kernel"], state["v"], state["L"], state["fmask"], state["vmapP"], state["s"], state["u"],
                       state["out"], accumulate=state["accumulate"])
    return lc.elementwise(state["kernel"], state["v"], state["arrays"], params=(0.7071,))


def work(case):
    """Each input read once, each output written once; multiply-adds as two operations."""
    op = case["op"]
    if op in ("contract", "geo"):
        E, N, F = case["E"], case["N"], case["F"]
        size = 8 if case["precision"] == "fp64" else 4
        values = E * N * (1 + F) + F * N * N + (E * F * F if op == "geo" else 0)
        return dict(bytes=size * values, flops=2 * E * N * N * F + (2 * E * N * F * F if op == "geo" else 0))
    if op == "grouped":
        F = case["F"]
        shapes = [(case[f"E{g}"], case[f"N{g}"]) for g in range(case["groups"])]
        return dict(bytes=sum(4 * (E * N * (1 + F) + F * N * N) for E, N in shapes),
                    flops=sum(2 * E * N * N * F for E, N in shapes))
    if op == "lift":
        E, p = case["E"], case["degree"]
        N, M = (p + 1) * (p + 2) * (p + 3) // 6, 2 * (p + 1) * (p + 2)
        return dict(bytes=4 * (E * (M + 4 + 2 * N) + N * M + M), flops=E * (2 * N * M + 2 * M))
    return dict(bytes=12 * case["n"], flops=2 * case["n"])


# ------------------------------------------------------------------ the same in 64 bits

def _contract64(D, u, layout):
    return torch.einsum("fij,je->fie" if layout == "node" else "fij,ej->fei", D.double(), u.double())


def exact(case, seed):
    """What run() returns for prepare(case, seed), in plain torch on float64."""
    gen = _gen(seed)
    op = case["op"]
    if op == "contract":
        D, u = _operands(gen, case["E"], case["N"], case["F"], case["layout"], case["precision"], case["scale"])
        return _contract64(D, u, case["layout"])
    if op == "grouped":
        outs = []
        for g in range(case["groups"]):
            D, u = _operands(gen, case[f"E{g}"], case[f"N{g}"], case["F"], case["layout"], case["precision"])
            outs.append(_contract64(D, u, case["layout"]))
        return outs
    if op == "geo":
        E, F, layout = case["E"], case["F"], case["layout"]
        D, u = _operands(gen, E, case["N"], F, layout, case["precision"])
        r = torch.randn((F, F, E) if layout == "node" else (E, F, F), generator=gen, device="cuda").double()
        part = _contract64(D, u, layout)
        return torch.einsum("dfe,fie->die" if layout == "node" else "edf,fei->dei", r, part)
    if op == "lift":
        E = case["E"]
        N, Nfp, fmask, vmapP = _mesh(E, case["degree"], case["width"])
        L = torch.rand((N, 4 * Nfp), generator=gen, device="cuda").mul_(2).sub_(1).double()
        s = torch.rand((E, 4), generator=gen, device="cuda").mul_(1.5).add_(0.5).double()
        u = torch.randn((E, N), generator=gen, device="cuda").double()
        jump = u[:, fmask.long()] - u.reshape(-1)[vmapP.long()]
        return (jump * s.repeat_interleave(Nfp, dim=1)) @ L.t()
    n = case["n"]
    x = torch.randn(n, generator=gen, device="cuda")
    y = torch.randn(n, generator=gen, device="cuda")
    a = float(torch.tensor(0.7071))  # the parameter is a binary32 value
    return x.double() * a + y.double()
