"""Direct contraction of tiny sectors (csrc/direct.cu): steps and chunks of its
streams at their edges, one to four columns a side, one to three box dims,
forward and gradients against the oracle, and the launch of both gradients
against the launches of one."""
import numpy as np
import pytest
import torch

from oracle import contract as oc
from oracle import u1 as ou1

pytestmark = pytest.mark.gpu

import paper_1203_2222_gb300 as P  # noqa: E402
from paper_1203_2222_gb300 import synthetic  # noqa: E402

# extents of the large operand's free legs (their product: positions of an
# item's stream, in steps of 256 down to 32, chunks of 1024 and 2048), its
# leg order, and the sizes of the contracted and of the other small leg
CASES = [((1, 1), "lxr", 1, 1), ((31, 1), "xlr", 1, 4), ((33, 1), "lrx", 4, 1), ((5, 13), "lxr", 2, 3),
         ((17, 15), "xrl", 4, 4), ((1023, 1), "lxr", 1, 1), ((41, 25), "rxl", 4, 4), ((32, 64), "lxr", 3, 2),
         ((43, 48), "rlx", 4, 4), ((7, 11, 29), "lxmr", 4, 4), ((9, 8, 5), "rmxl", 2, 4), ((6, 7, 50), "mlrx", 1, 3)]


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("ext,order,k,n", CASES)
def test_direct_against_the_oracle(ext, order, k, n, dtype):
    q = [0, 1]
    legs = {"l": (q, [ext[0], 3], 1), "m": (q, [ext[1], 2], 1), "r": (q, [ext[-1], 5], -1), "x": (q, [k, 1], -1)}
    la = [legs[c] for c in order]
    lb = [(q, [k, 1], 1), (q, [n, 2], -1)]
    pa, pb = [order.index("x")], [0]
    SA, SB = P.Structure(P.U1, la), P.Structure(P.U1, lb)
    a = P.SymTensor.from_numpy(SA, synthetic.normal(1, SA.numel), dtype=dtype)
    b = P.SymTensor.from_numpy(SB, synthetic.normal(2, SB.numel), dtype=dtype)
    a.data.requires_grad_(True)
    b.data.requires_grad_(True)
    C = P.contract(a, b, pa, pb)
    g = torch.as_tensor(synthetic.normal(3, C.structure.numel)).to(dtype).cuda()
    da, db = torch.autograd.grad(C.data, [a.data, b.data], grad_outputs=g, retain_graph=True)
    oa = ([ou1.Leg(*l) for l in la], 0, a.data.detach().double().cpu().numpy())
    ob = ([ou1.Leg(*l) for l in lb], 0, b.data.detach().double().cpu().numpy())
    _, _, c_ref, _ = oc.contract("u1", oa, ob, pa, pb)
    da_ref, db_ref, _ = oc.contract_grad("u1", oa, ob, pa, pb, g.double().cpu().numpy())
    # random terms: a rounding error per term grows like the square root of their number
    eps = 1.2e-7 if dtype == torch.float32 else 2.3e-16
    for x, ref, terms in ((C.data.detach(), c_ref, k), (da, da_ref, n), (db, db_ref, int(np.prod(ext)))):
        x = x.double().cpu().numpy()
        assert np.linalg.norm(x - ref) <= eps * (4.0 + np.sqrt(terms)) * np.linalg.norm(ref)
    (da1,) = torch.autograd.grad(C.data, [a.data], grad_outputs=g, retain_graph=True)
    (db1,) = torch.autograd.grad(C.data, [b.data], grad_outputs=g)
    assert torch.equal(da, da1)  # the same sums in the same order
    # sums of the same terms in two orders of their parts
    assert float((db - db1).norm()) <= 2 * eps * (4.0 + np.sqrt(np.prod(ext))) * float(db.norm())
    torch.cuda.synchronize()
    P.device_status()
