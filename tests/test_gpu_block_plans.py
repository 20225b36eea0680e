"""Contractions on the blocks (csrc/block.cu) whose plans are checked first: each
tile shape, reductions cut into parts (launched again and again: the arrival
counters return to zero), more pairs of blocks than the kernel keeps in shared
memory, and batches that mix blocks and matrix form."""
import numpy as np
import pytest
import torch

from oracle import contract as oc
from oracle import u1 as ou1

pytestmark = pytest.mark.gpu

import paper_1203_2222_gb300 as P  # noqa: E402
from paper_1203_2222_gb300 import synthetic  # noqa: E402

PREC = {torch.float32: P.BF16X3, torch.float64: P.FP64}


def _matrix(m, n, k):
    q = [0, 1]
    mid = [k, max(1, k // 2)]
    return [(q, [m, max(1, m // 3)], 1), (q, mid, -1)], [(q, mid, 1), (q, [n, max(1, n // 5)], -1)], [1], [0]


def _many_segments(f):
    """31 pairs of blocks meet in an output block (24 of them are kept in shared memory)."""
    q = list(range(-15, 16))
    con = [(q, [2] * 31, 1), (q, [1] * 31, -1)]
    return (con + [([-1, 0, 1], [f, f + 1, f], 1)],
            [(l, d, -s) for l, d, s in con] + [([-1, 0, 1], [f + 2, f, 1], 1)], [0, 1], [0, 1])


F32, F64 = torch.float32, torch.float64
# (legs, type, shapes the plan has to use, whether it has to cut a reduction, pairs of blocks a tile)
CASES = {
    "large, cut dots": (_matrix(12, 12, 4000), F32, ("large", "medium", "small", "tall", "dot"), True, 1),
    "dots in parts": (_matrix(5, 8, 30000), F32, ("tall", "dot"), True, 1),
    "dots in parts, FP64": (_matrix(5, 8, 30000), F64, ("tall", "dot"), True, 1),
    "medium and small in parts": (_matrix(70, 70, 3000), F32, ("medium", "small"), True, 1),
    "small in parts, FP64": (_matrix(70, 70, 3000), F64, ("small",), True, 1),
    "medium in parts, FP64": (_matrix(40, 40, 20000), F64, ("medium", "small", "tall"), True, 1),
    "tall in parts, FP64": (_matrix(300, 6, 40), F64, ("small", "tall"), True, 1),
    "31 segments": (_many_segments(3), F32, ("small",), False, 31),
    "31 segments, FP64": (_many_segments(3), F64, ("small",), False, 31),
    "31 segments in parts, FP64": (_many_segments(20), F64, ("medium", "small", "tall"), True, 31),
}


def _oracle(la, lb, pa, pb, a, b, g):
    oa, ob = ([ou1.Leg(*l) for l in la], 0, a), ([ou1.Leg(*l) for l in lb], 0, b)
    _, _, c, _ = oc.contract("u1", oa, ob, pa, pb)
    da, db, _ = oc.contract_grad("u1", oa, ob, pa, pb, g)
    return c, da, db


def _rel(x, ref):
    x = x.detach().double().cpu().numpy()
    return float(np.linalg.norm(x - ref) / max(np.linalg.norm(ref), 1e-300))


def _data(n, seed, dtype):
    return torch.as_tensor(synthetic.normal(seed, n)).to(dtype).cuda()


def _bound(dtype, terms):  # a rounding error per step of a sum grows like the square root of their number
    return (1.2e-7 if dtype == F32 else 2.3e-16) * (4.0 + np.sqrt(terms))


@pytest.mark.parametrize("name", sorted(CASES))
def test_planned_shapes_against_the_oracle(name):
    (la, lb, pa, pb), dtype, shapes, cut, segments = CASES[name]
    SA, SB = P.Structure(P.U1, la), P.Structure(P.U1, lb)
    plan = P.contract_plan(SA, SB, pa, pb, PREC[dtype])
    info = plan.block_info()
    assert all(info["tiles"][s] for s in shapes), info
    assert (info["cut"] > 0) == cut and info["segments"] == segments, info
    a, b = _data(SA.numel, 1, dtype), _data(SB.numel, 2, dtype)
    a.requires_grad_(True), b.requires_grad_(True)
    g = _data(plan.out.numel, 3, dtype)
    plan.profile(True)
    runs = []
    for _ in range(4):
        c = P.contract(P.SymTensor(SA, a), P.SymTensor(SB, b), pa, pb).data
        runs.append((c.detach(),) + torch.autograd.grad(c, [a, b], grad_outputs=g))
    torch.cuda.synchronize()
    plan.profile(False)
    P.device_status()
    launches = {k: plan.profile_kernel(i)["launches"] for k, i in P.KERNELS.items()}
    assert launches["block"] == 2 * len(runs) == sum(launches.values())
    for r in runs[1:]:
        assert all(torch.equal(x, y) for x, y in zip(r, runs[0]))
    ref = _oracle(la, lb, pa, pb, *(x.detach().double().cpu().numpy() for x in (a, b, g)))
    terms = max(max(d) for _, d, _ in la + lb)
    for x, y in zip(runs[0], ref):
        assert _rel(x, y) <= _bound(dtype, terms)


@pytest.mark.parametrize("dtype", [F32, F64])
def test_batch_of_blocks_and_matrix_form(dtype):
    sizes = [(8, 8, 60000), (40, 30, 9), (600, 500, 300), (8, 300000, 3)]
    legs = [_matrix(m, n, k) for m, n, k in sizes]
    SA, SB = [P.Structure(P.U1, l[0]) for l in legs], [P.Structure(P.U1, l[1]) for l in legs]
    plan = P.contract_batch_plan(SA, SB, [1], [0], PREC[dtype])
    info = plan.block_info()
    assert sum(info["tiles"].values()) > 0 and info["workspace"] <= 64 << 20
    assert (dtype == F64) or info["cut"] > 0  # FP64: the other problems fill the launch
    a, b = _data(plan.off_a[-1], 1, dtype), _data(plan.off_b[-1], 2, dtype)
    a.requires_grad_(True), b.requires_grad_(True)
    g = _data(plan.off_c[-1], 3, dtype)
    plan.profile(True)
    for _ in range(3):
        c = P.contract_batch(plan, a, b)
        da, db = torch.autograd.grad(c, [a, b], grad_outputs=g)
    torch.cuda.synchronize()
    plan.profile(False)
    P.device_status()
    launches = {k: plan.profile_kernel(i)["launches"] for k, i in P.KERNELS.items()}
    assert launches["block"] == 6
    if dtype == F32:
        assert launches["gemm_tc"] > 0
    for i, (la, lb, pa, pb) in enumerate(legs):
        sl = [slice(o[i], o[i + 1]) for o in (plan.off_a, plan.off_b, plan.off_c)]
        x = [t.detach().double().cpu().numpy() for t in (a[sl[0]], b[sl[1]], g[sl[2]])]
        for got, ref in zip((c[sl[2]], da[sl[0]], db[sl[1]]), _oracle(la, lb, pa, pb, *x)):
            # split-BF16: 3 * 2^-17 of every product
            assert _rel(got, ref) <= (2e-5 if dtype == F32 else _bound(dtype, 3e5))
