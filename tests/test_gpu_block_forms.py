"""Which form a contraction runs in (csrc/plan.cpp): on the blocks, or in
matrix form while its stream is captured, with every mix of captured and plain
calls against the oracle."""
import numpy as np
import pytest
import torch

from oracle import contract as oc
from oracle import u1 as ou1
from tests.graph_replay import replay

pytestmark = pytest.mark.gpu

import paper_1203_2222_gb300 as P  # noqa: E402
from paper_1203_2222_gb300 import _lib as lib  # noqa: E402
from paper_1203_2222_gb300 import synthetic  # noqa: E402


def _chain(D, qmax):
    """L.A of a U(1) chain: structures, legs and plan (FP32)."""
    w = synthetic.u1_mps_heff(D=D, qmax=qmax, sigma=0.3 * qmax)
    L, A = P.Structure(P.U1, w["L"]), P.Structure(P.U1, w["A"])
    return w, L, A, P.contract_plan(L, A, [2], [0], P.BF16X3)


def _rel(x, ref):
    x = x.detach().double().cpu().numpy()
    return float(np.linalg.norm(x - ref) / np.linalg.norm(ref))


# few sectors large enough for the tensor cores: the blocks win by the launches alone
@pytest.mark.parametrize("D,qmax", [(400, 3), (600, 3)])
def test_captured_and_plain_calls_mixed(D, qmax):
    w, SL, SA, plan = _chain(D, qmax)
    oL, oA = (([ou1.Leg(*l) for l in w[n]], 0, synthetic.normal(i, S.numel))
              for i, (n, S) in enumerate((("L", SL), ("A", SA))))
    _, _, c_ref, _ = oc.contract("u1", oL, oA, [2], [0])
    g_np = synthetic.normal(3, plan.out.numel)
    da_ref, db_ref, _ = oc.contract_grad("u1", oL, oA, [2], [0], g_np)
    a, b, g = (torch.as_tensor(x).float().cuda() for x in (oL[2], oA[2], g_np))
    c, da, db = torch.empty_like(g), torch.empty_like(a), torch.empty_like(b)

    def forward():
        lib.check(lib.lib.sym_contract(plan._h, a.data_ptr(), b.data_ptr(), c.data_ptr(),
                                       torch.cuda.current_stream().cuda_stream))

    def backward():
        lib.check(lib.lib.sym_contract_backward(plan._h, a.data_ptr(), b.data_ptr(), g.data_ptr(), da.data_ptr(),
                                                db.data_ptr(), torch.cuda.current_stream().cuda_stream))

    def run(*steps):
        """Each step plain or captured, in order; the inputs are in place only when the graphs run."""
        graphs = []
        for fn, captured in steps:
            if captured:
                a.mul_(2.0)
                graphs.append(replay(fn, warmup=0)[1])
                a.div_(2.0)
        for x in (c, da, db):
            x.fill_(float("nan"))
        it = iter(graphs)
        for fn, captured in steps:
            next(it).replay() if captured else fn()
        torch.cuda.synchronize()
        P.device_status()
        for x, ref in ((c, c_ref), (da, da_ref), (db, db_ref)):
            assert _rel(x, ref) <= 2e-5  # split-BF16: 3 * 2^-17 of every product

    plan.profile(True)
    run((forward, False), (backward, False))
    plan.profile(False)
    k = {name: plan.profile_kernel(i)["launches"] for name, i in P.KERNELS.items()}
    assert k["block"] == 2 and sum(k.values()) == 2
    run((forward, True), (backward, True))
    run((lambda: (forward(), backward()), True))
    run((forward, False), (backward, True))
    run((forward, True), (backward, False))


def test_the_captured_form_is_the_matrix_form():
    _, SL, SA, plan = _chain(600, 3)
    a, b = torch.randn(SL.numel, device="cuda"), torch.randn(SA.numel, device="cuda")
    replay(lambda: P.contract(P.SymTensor(SL, a), P.SymTensor(SA, b), [2], [0]).data)  # warm
    plan.profile(True)
    s = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=s):
        P.contract(P.SymTensor(SL, a), P.SymTensor(SA, b), [2], [0])
    n_captured = plan.launches()
    plan.profile(False)
    graph.replay()
    torch.cuda.synchronize()
    k = {name: plan.profile_kernel(i)["launches"] for name, i in P.KERNELS.items()}
    assert k["block"] == 0 and k["gemm_tc"] == 1 and n_captured == sum(k.values())
