"""Contractions that run on the tensors' blocks (csrc/block.cu): every tile
shape at its edges against the oracle, and random leg orders against the
matrix-form path, forward and both gradients."""
import numpy as np
import pytest
import torch

from oracle import contract as oc
from oracle import u1 as ou1
from oracle import z2f as oz

pytestmark = pytest.mark.gpu

import paper_1203_2222_gb300 as P  # noqa: E402
from paper_1203_2222_gb300 import synthetic  # noqa: E402


def _run(group, la, lb, pa, pb, dtype, seed):
    SA, SB = P.Structure(group, la), P.Structure(group, lb)
    a = P.SymTensor.from_numpy(SA, synthetic.normal(seed, SA.numel), dtype=dtype)
    b = P.SymTensor.from_numpy(SB, synthetic.normal(seed + 1, SB.numel), dtype=dtype)
    a.data.requires_grad_(True)
    b.data.requires_grad_(True)
    C = P.contract(a, b, pa, pb)
    g = torch.as_tensor(synthetic.normal(seed + 2, C.structure.numel)).to(dtype).cuda()
    da, db = torch.autograd.grad(C.data, [a.data, b.data], grad_outputs=g)
    torch.cuda.synchronize()
    P.device_status()
    return a.data.detach(), b.data.detach(), g, C.data.detach(), da, db


def _rel(x, ref):
    x, ref = x.double().cpu().numpy(), np.asarray(ref)
    return float(np.linalg.norm(x - ref) / max(np.linalg.norm(ref), 1e-300))


# (m, n, k) of the charge-0 blocks around the tile and slab edges: 8 x 8 outputs
# with long reductions (and their parts), narrow outputs, 32, 48 and 64 wide tiles
SIZES = [(1, 1, 1), (1, 1, 20000), (8, 8, 700), (9, 8, 513), (257, 7, 9), (31, 33, 15), (32, 32, 32), (47, 49, 17),
         (65, 63, 33), (129, 127, 16), (200, 48, 5), (7, 300, 40), (70, 70, 3000)]


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("m,n,k", SIZES)
def test_tile_edges_against_the_oracle(m, n, k, dtype):
    q = [0, 1]
    la = [(q, [m, max(1, m // 3)], 1), (q, [k, max(1, k // 2)], -1)]
    lb = [(q, [k, max(1, k // 2)], 1), (q, [n, max(1, n // 5)], -1)]
    a, b, g, c, da, db = _run(P.U1, la, lb, [1], [0], dtype, 100)
    oa = ([ou1.Leg(*l) for l in la], 0, a.double().cpu().numpy())
    ob = ([ou1.Leg(*l) for l in lb], 0, b.double().cpu().numpy())
    _, _, c_ref, _ = oc.contract("u1", oa, ob, [1], [0])
    da_ref, db_ref, _ = oc.contract_grad("u1", oa, ob, [1], [0], g.double().cpu().numpy())
    # random terms summed in order: a rounding error per step grows like the square root of their number
    eps = 1.2e-7 if dtype == torch.float32 else 2.3e-16
    for x, ref, terms in ((c, c_ref, k), (da, da_ref, n), (db, db_ref, m)):
        assert _rel(x, ref) <= eps * (4.0 + np.sqrt(terms))


@pytest.mark.parametrize("group", ["u1", "z2f", "su2", "su2u1"])
@pytest.mark.parametrize("seed", range(6))
def test_any_leg_order_matches_the_matrix_form(group, seed):
    rng = np.random.default_rng(seed)
    g = {"u1": P.U1, "z2f": P.Z2F, "su2": P.SU2, "su2u1": P.SU2U1}[group]
    labels = {"u1": [-1, 0, 1], "z2f": [0, 1], "su2": [0, 1, 2], "su2u1": [(-1, 1), (0, 0), (1, 1)]}[group]
    nc, na, nb = int(rng.integers(1, 3)), int(rng.integers(1, 3)), int(rng.integers(1, 3))

    def leg():
        return (labels, [int(x) for x in rng.integers(1, 9, len(labels))], int(rng.choice([-1, 1])))

    con = [leg() for _ in range(nc)]
    A, B = con + [leg() for _ in range(na)], [(l, d, -s) for l, d, s in con] + [leg() for _ in range(nb)]
    oa, ob = rng.permutation(nc + na), rng.permutation(nc + nb)
    la, lb = [A[i] for i in oa], [B[i] for i in ob]
    pa, pb = [int(np.where(oa == i)[0][0]) for i in range(nc)], [int(np.where(ob == i)[0][0]) for i in range(nc)]
    if not (P.Structure(g, la).numel and P.Structure(g, lb).numel):
        pytest.skip("no block")
    got = _run(g, la, lb, pa, pb, torch.float64, 10 * seed)
    tune = P.tune_get()
    try:
        P.tune_set(tc_min_mn=65)  # a kernel choice of its own: every phase in matrix form
        ref = _run(g, la, lb, pa, pb, torch.float64, 10 * seed)
    finally:
        P.tune_set(**tune)
    for x, y in zip(got[3:], ref[3:]):
        assert _rel(x, y.cpu().numpy()) <= 1e-13


def test_fermion_signs_against_the_oracle():
    la = [([0, 1], [5, 9], 1), ([0, 1], [7, 3], -1), ([0, 1], [4, 6], 1), ([0, 1], [8, 5], -1)]
    lb = [([0, 1], [8, 5], 1), ([0, 1], [33, 34], 1), ([0, 1], [7, 3], 1)]
    a, b, g, c, da, db = _run(P.Z2F, la, lb, [3, 1], [0, 2], torch.float64, 7)
    oa = ([oz.Leg(*l) for l in la], 0, a.cpu().numpy())
    ob = ([oz.Leg(*l) for l in lb], 0, b.cpu().numpy())
    _, _, c_ref, _ = oc.contract("z2f", oa, ob, [3, 1], [0, 2])
    assert _rel(c, c_ref) <= 1e-14
