"""The FP64 refinement of the blockwise SVD and eigendecomposition
(csrc/svd.cu): blocks at the edges of its tiles and of the FP32 sweeps by
column blocks, of less than full rank, with equal or signed-equal values,
tall and wide, against numpy."""
import numpy as np
import pytest
import torch

import paper_1203_2222_gb300 as P
from paper_1203_2222_gb300 import synthetic

pytestmark = pytest.mark.gpu


def _mat(n, m, seed):
    return synthetic.normal(seed, n * m).reshape(n, m)


def _orth(n, seed):
    return np.linalg.qr(_mat(n, n, seed))[0]


def _two_blocks(M):
    """U(1) tensor with M as its charge-0 block and a small random charge-1 block."""
    n, m = M.shape
    S = P.Structure(P.U1, [([0, 1], [n, 3], 1), ([0, 1], [m, 5], -1)])
    pos, off = S.sectors()
    v = synthetic.normal(5, S.numel)
    for s in range(S.nsec):
        if S.legs[0][0][pos[s][0]] == 0:
            v[off[s]:off[s + 1]] = M.reshape(-1)
    return S, torch.as_tensor(v).cuda()


SVD = {
    "1x1": lambda: _mat(1, 1, 1), "31": lambda: _mat(31, 31, 2), "33x32": lambda: _mat(33, 32, 3),
    "63": lambda: _mat(63, 63, 4), "64x65": lambda: _mat(64, 65, 5), "tall 385x70": lambda: _mat(385, 70, 6),
    "wide 64x641": lambda: _mat(64, 641, 7), "tall 640x66": lambda: _mat(640, 66, 8),
    "rank 20 of 70": lambda: _mat(70, 20, 9) @ _mat(20, 70, 10), "rank 1": lambda: _mat(40, 1, 11) @ _mat(1, 40, 12),
    "zero": lambda: np.zeros((40, 33)), "zero columns": lambda: np.pad(_mat(50, 20, 13), ((0, 0), (0, 15))),
    "orthogonal": lambda: _orth(70, 14), "diagonal": lambda: np.diag(synthetic.normal(15, 70)),
    "graded": lambda: (_orth(70, 16) * np.logspace(0, -20, 70)) @ _orth(70, 17),
    "tiny": lambda: 1e-150 * _mat(40, 40, 18), "huge": lambda: 1e150 * _mat(40, 40, 19),
}


# FP32 sweeps through Gram matrices: each width of a column block (2 .. 14), the
# last blocks ragged or absent, and rows that are no multiple of a warp's
SVD.update({f"blocks of {b}": lambda b=b: _mat(32 * b - 31 + 3 * b, 32 * b - 31, 30 + b) for b in range(3, 15)})
SVD["blocks of 2"] = lambda: _mat(64, 64, 31)
SVD["blocks of 14, full"] = lambda: _mat(448, 448, 32)
SVD["blocks of 5, rows past their shared memory"] = lambda: _mat(2600, 160, 33)


@pytest.mark.parametrize("name", sorted(SVD))
def test_svd(name):
    M = SVD[name]()
    S, v = _two_blocks(M)
    U, s, V = P.svd(P.SymTensor(S, v), 1)
    torch.cuda.synchronize()
    P.device_status()
    n, m = M.shape
    k = min(n, m)
    # block 0 leads in U, V and the values (the first leg is outgoing)
    u = U.data[:n * k].cpu().numpy().reshape(n, k)
    w = V.data[:k * m].cpu().numpy().reshape(k, m)
    s = s[:k].cpu().numpy()
    ref = np.linalg.svd(M, compute_uv=False)
    scale = max(ref[0], 1e-300)
    assert np.max(np.abs(s - ref)) <= 1e-12 * scale
    assert np.linalg.norm(((u * (s / scale)) @ w) - M / scale) <= 1e-12 * max(np.sqrt(k), 1.0)
    assert np.max(np.abs(w @ w.T - np.eye(k))) <= 1e-12 or s[-1] == 0.0
    live = s > 1e-10 * scale  # vectors of zero values are zeros where they come from a division
    g = u[:, live].T @ u[:, live]
    assert np.max(np.abs(g - np.eye(g.shape[0])), initial=0.0) <= 1e-12


EIG = {
    "3": lambda: _mat(3, 3, 1), "33": lambda: _mat(33, 33, 2), "65": lambda: _mat(65, 65, 3),
    "psd rank 20 of 70": lambda: _mat(70, 20, 4) @ _mat(70, 20, 4).T,
    "psd full": lambda: _mat(70, 75, 5) @ _mat(70, 75, 5).T, "zero": lambda: np.zeros((33, 33)),
    "signs": lambda: (_orth(66, 6) * np.sign(synthetic.normal(7, 66))) @ _orth(66, 6).T,
    "clusters": lambda: (_orth(66, 8) * np.repeat([2.0, -1.0, 1e-3], 22)) @ _orth(66, 8).T,
    "negative": lambda: -_mat(65, 70, 9) @ _mat(65, 70, 9).T, "tiny": lambda: 1e-150 * _mat(40, 40, 10),
}


@pytest.mark.parametrize("name", sorted(EIG))
def test_eig(name):
    M = EIG[name]()
    M = 0.5 * (M + M.T)
    n = M.shape[0]
    S = P.Structure(P.U1, [([0], [n], 1), ([0], [n], -1)])
    U, lam, V = P.eig(P.SymTensor(S, torch.as_tensor(M.reshape(-1)).cuda()), 1)
    torch.cuda.synchronize()
    P.device_status()
    u, lam = U.data.cpu().numpy().reshape(n, n), lam.cpu().numpy()
    ref = np.linalg.eigvalsh(M)
    scale = max(np.max(np.abs(ref)), 1e-300)
    assert np.max(np.abs(np.sort(lam) - ref)) <= 1e-12 * scale
    assert np.all(np.diff(np.abs(lam)) <= 1e-12 * scale)
    assert np.max(np.abs(u.T @ u - np.eye(n))) <= 1e-12
    assert np.linalg.norm((M / scale) @ u - u * (lam / scale)) <= 1e-12 * np.sqrt(n)
    np.testing.assert_array_equal(V.data.cpu().numpy().reshape(n, n), u.T)
