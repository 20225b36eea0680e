"""Blockwise SVD and eigendecomposition (csrc/svd.cu) of blocks whose columns
or whose values lie far from 1: the angles of the FP32 sweeps, the norms and
the levels of the refinement keep their ratios at every scale."""
import numpy as np
import pytest
import torch

import paper_1203_2222_gb300 as P
from paper_1203_2222_gb300 import synthetic

pytestmark = pytest.mark.gpu


def _mat(n, m, seed):
    return synthetic.normal(seed, n * m).reshape(n, m)


def _svd(M):
    """(u, s, w) of one block on the GPU."""
    n, m = M.shape
    k = min(n, m)
    S = P.Structure(P.U1, [([0], [n], 1), ([0], [m], -1)])
    U, s, V = P.svd(P.SymTensor(S, torch.as_tensor(np.ascontiguousarray(M).reshape(-1)).cuda()), 1)
    torch.cuda.synchronize()
    P.device_status()
    return U.data.cpu().numpy().reshape(n, k), s.cpu().numpy(), V.data.cpu().numpy().reshape(k, m)


def _pairs_of_tiny_columns(n, e):
    """One entry 1; the other columns random, e times as large, and two of them equal."""
    M = np.zeros((n, n))
    M[0, 0] = 1.0
    M[1:, 1:] = e * _mat(n - 1, n - 1, 77)
    M[1:, 2] = M[1:, 1]
    return M


# e^2 is still a normal FP32 number for the first three, e^4 for the first one
# only; n: the sweeps by pairs and through Gram matrices
@pytest.mark.parametrize("e", [1e-8, 1e-11, 1e-13, 1e-18])
@pytest.mark.parametrize("n", [3, 40, 70])
def test_svd_with_equal_tiny_columns(n, e):
    M = _pairs_of_tiny_columns(n, e)
    u, s, w = _svd(M)
    ref = np.linalg.svd(M, compute_uv=False)
    # the values next to 1 to FP64 accuracy of e: the columns' own scale
    assert abs(s[0] - 1.0) <= 1e-14
    assert np.max(np.abs(s[1:] - ref[1:])) <= 1e-12 * e * np.sqrt(n)
    assert np.max(np.abs(w @ w.T - np.eye(n))) <= 1e-12
    assert np.max(np.abs((u * s) @ w - M)[1:, 1:]) <= 1e-12 * e * np.sqrt(n)


@pytest.mark.parametrize("n", [39, 40, 41, 70])
def test_svd_with_one_entry_far_above_the_others(n):
    # scaled by any entry but the largest, the block is out of FP32's range (several
    # runs: which CTA of the cluster finds the largest entry last is not fixed)
    e = 1e-60
    for seed in range(8):
        M = e * _mat(n, n, seed)
        M[seed % n, (3 * seed) % n] = 1.0
        u, s, w = _svd(M)
        assert abs(s[0] - 1.0) <= 1e-14 and np.all(np.abs(s[1:]) <= 1e-14)
        assert np.max(np.abs(w @ w.T - np.eye(n))) <= 1e-12
        assert np.linalg.norm((u * s) @ w - M) <= 1e-14


def _eig(M):
    n = M.shape[0]
    S = P.Structure(P.U1, [([0], [n], 1), ([0], [n], -1)])
    U, lam, _ = P.eig(P.SymTensor(S, torch.as_tensor(np.ascontiguousarray(M).reshape(-1)).cuda()), 1)
    torch.cuda.synchronize()
    P.device_status()
    return U.data.cpu().numpy().reshape(n, n), lam.cpu().numpy()


# squares of the values over- and underflow beyond 1e+-154; the same block scaled by a
# power of two has the same factors, and values that differ by that power alone
@pytest.mark.parametrize("power", [-1000, -660, -531, -520, -512, 512, 531, 660, 1000])
@pytest.mark.parametrize("n", [2, 40, 70])
def test_values_whose_squares_leave_the_range(n, power):
    M = _mat(n, n + 1, 18)
    u, s, w = _svd(M)
    u2, s2, w2 = _svd(np.ldexp(M, power))
    np.testing.assert_array_equal(np.ldexp(s2, -power), s)
    np.testing.assert_array_equal(u2, u)
    np.testing.assert_array_equal(w2, w)
    B = _mat(n, n, 10)
    B = 0.5 * (B + B.T)
    q, lam = _eig(B)
    q2, lam2 = _eig(np.ldexp(B, power))
    np.testing.assert_array_equal(np.ldexp(lam2, -power), lam)
    np.testing.assert_array_equal(q2, q)
    ref = np.linalg.eigvalsh(B)
    assert np.linalg.norm(B @ q - q * lam) <= 1e-12 * np.sqrt(n) * np.max(np.abs(ref))
    assert np.max(np.abs(np.sort(lam) - ref)) <= 1e-12 * np.max(np.abs(ref))


@pytest.mark.parametrize("e", [1e-16, 1e-20, 1e-25, 1e-45, 1e-60])
@pytest.mark.parametrize("n", [5, 40, 70])
def test_svd_with_one_tiny_column(n, e):
    M = _mat(n, n, 21)
    M[:, n - 1] *= e
    u, s, w = _svd(M)
    # the value of the tiny column: what the other columns do not span of it
    Q, _ = np.linalg.qr(M[:, :n - 1])
    x = M[:, n - 1] / e
    x -= Q @ (Q.T @ x)
    x -= Q @ (Q.T @ x)
    assert abs(s[-1] / e - np.linalg.norm(x)) <= 1e-12 * np.linalg.norm(M) / np.min(s[:-1])
    assert np.max(np.abs(u.T @ u - np.eye(n))) <= 1e-12
    assert np.max(np.abs(w @ w.T - np.eye(n))) <= 1e-12


@pytest.mark.parametrize("e", [1.0, 1e-8, 1e-11, 1e-13, 1e-18])
@pytest.mark.parametrize("n", [5, 40, 70])
def test_svd_with_equal_rows(n, e):
    # one entry 1, all others in the rest equal: every column of A V that belongs to a
    # zero value is rounding, and an exact multiple of every other
    M = np.zeros((n, n))
    M[0, 0] = 1.0
    M[1:, 1:] = e
    u, s, w = _svd(M)
    ref = sorted([1.0, e * (n - 1)], reverse=True)
    assert np.max(np.abs(s[:2] / ref - 1.0)) <= 1e-14
    assert np.all(np.abs(s[2:]) <= n * 2.3e-16 * ref[0])
    assert np.max(np.abs(w @ w.T - np.eye(n))) <= 1e-12
    assert np.max(np.abs(u[:, :2].T @ u[:, :2] - np.eye(2))) <= 1e-12
    assert np.max(np.abs((u * s) @ w - M)[1:, 1:]) <= 1e-14 * e * n


def _orth(n, seed):
    return np.linalg.qr(_mat(n, n, seed))[0]


DECAYS = {f"1e-{d}": lambda n, d=d: np.logspace(0, -d, n) for d in (4, 6, 8, 10, 14, 20)}
DECAYS.update({f"k^-{p}": lambda n, p=p: np.arange(1.0, n + 1.0) ** -p for p in (4, 6, 8)})
DECAYS["signs"] = lambda n: np.logspace(0, -9, n) * (-1.0) ** np.arange(n)
DECAYS["gaps of 1e-9"] = lambda n: 1.0 + 1e-9 * np.arange(n)
DECAYS["gaps of 1e-11"] = lambda n: 1.0 + 1e-11 * np.arange(n)


@pytest.mark.parametrize("name", sorted(DECAYS))
@pytest.mark.parametrize("n", [40, 70, 128])
def test_close_and_decaying_values(n, name):
    v = DECAYS[name](n)
    Q = _orth(n, 7)
    B = (Q * v) @ Q.T
    B = 0.5 * (B + B.T)
    q, lam = _eig(B)
    assert np.linalg.norm(B @ q - q * lam) <= 1e-12 * np.sqrt(n)
    assert np.max(np.abs(np.sort(lam) - np.linalg.eigvalsh(B))) <= 1e-12
    assert np.max(np.abs(q.T @ q - np.eye(n))) <= 1e-12
    M = (_orth(n, 5) * v) @ _orth(n, 6)
    u, s, w = _svd(M)
    assert np.linalg.norm((u * s) @ w - M) <= 1e-12 * np.sqrt(n)
    assert np.max(np.abs(s - np.linalg.svd(M, compute_uv=False))) <= 1e-12
    assert np.max(np.abs(w @ w.T - np.eye(n))) <= 1e-12
    live = s > 1e-10 * s[0]
    assert np.max(np.abs(u[:, live].T @ u[:, live] - np.eye(live.sum()))) <= 1e-12


def test_workspace_is_bounded():
    """7.5 n^2 doubles a square block: V and W are refined where they are."""
    n = 3000
    S = P.Structure(P.U1, [([0], [n], 1), ([0], [n], -1)])
    P.svd_plan(P.Structure(P.U1, [([0], [8], 1), ([0], [8], -1)]), 1)  # whatever a first plan sets up
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    plan = P.svd_plan(S, 1)
    assert free - torch.cuda.mem_get_info()[0] <= 8.4 * n * n * 8
    del plan
