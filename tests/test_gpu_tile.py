"""The FP32 tile GEMM (csrc/gemm_simt.cu) at the edges of its tiles, warps and
slices, its two shapes and split reductions, forward and both gradients
against the oracle."""
import numpy as np
import pytest
import torch

from oracle import contract as oc
from oracle import u1 as ou1

pytestmark = pytest.mark.gpu

import paper_1203_2222_gb300 as P  # noqa: E402
from paper_1203_2222_gb300 import synthetic  # noqa: E402

# 64 x 64 tiles of 32 x 32 parts with slices of 16; 256 x 16 tiles of 64 x 16
# parts with slices of 8; reductions long enough to be split
SIZES = [(17, 17, 17), (31, 33, 15), (32, 32, 16), (33, 65, 47), (64, 64, 48), (65, 129, 33), (96, 20, 100),
         (63, 61, 3000), (255, 16, 17), (257, 11, 23), (64, 16, 24), (513, 9, 40), (20, 12, 5000), (300, 300, 31)]


@pytest.mark.parametrize("m,n,k", SIZES)
def test_tiles_against_the_oracle(m, n, k):
    q = [0, 1]
    la = [(q, [m, max(9, m // 3)], 1), (q, [k, max(17, k // 2)], -1)]
    lb = [(q, [k, max(17, k // 2)], 1), (q, [n, max(9, n // 2)], -1)]
    tune = P.tune_get()
    try:
        P.tune_set(tc_min_mn=1 << 20)  # matrix form, no sector on the tensor cores
        SA, SB = P.Structure(P.U1, la), P.Structure(P.U1, lb)
        a = P.SymTensor.from_numpy(SA, synthetic.normal(1, SA.numel), dtype=torch.float32)
        b = P.SymTensor.from_numpy(SB, synthetic.normal(2, SB.numel), dtype=torch.float32)
        a.data.requires_grad_(True)
        b.data.requires_grad_(True)
        C = P.contract(a, b, [1], [0])
        g = torch.as_tensor(synthetic.normal(3, C.structure.numel)).float().cuda()
        da, db = torch.autograd.grad(C.data, [a.data, b.data], grad_outputs=g)
        torch.cuda.synchronize()
        P.device_status()
    finally:
        P.tune_set(**tune)
    oa = ([ou1.Leg(*l) for l in la], 0, a.data.detach().double().cpu().numpy())
    ob = ([ou1.Leg(*l) for l in lb], 0, b.data.detach().double().cpu().numpy())
    _, _, c_ref, _ = oc.contract("u1", oa, ob, [1], [0])
    da_ref, db_ref, _ = oc.contract_grad("u1", oa, ob, [1], [0], g.double().cpu().numpy())
    # random terms summed in order: a rounding error per step grows like the square root of their number
    for x, ref, terms in ((C.data.detach(), c_ref, k), (da, da_ref, n), (db, db_ref, m)):
        x = x.double().cpu().numpy()
        assert np.linalg.norm(x - ref) <= 1.2e-7 * (4.0 + np.sqrt(terms)) * np.linalg.norm(ref)
