"""The block Jacobi eigensolver through the Rayleigh-Ritz step: orders around its
16-wide block pairs, clustered and degenerate spectra, extreme scales, NaN."""
import numpy as np
import pytest

import fd_inputs
from oracle import matrices as mat

pytestmark = pytest.mark.gpu


def _ritz(csr, V0):
    import torch

    import paper_2209_01974_gb300 as fd
    ctx = fd.fd_create(0)
    A = fd.fd_matrix_from_csr(ctx, *csr)
    V = torch.from_numpy(V0).cuda()
    AV = torch.empty_like(V)
    theta, resid = fd.fd_rayleigh_ritz(ctx, A, V, AV)
    return theta, resid, V.cpu().numpy()


def _check(csr, ns, seed):
    A = mat.to_scipy(csr)
    V0 = np.linalg.qr(fd_inputs.random_block(A.shape[0], ns, seed))[0]
    theta, resid, V = _ritz(csr, V0)
    H = V0.T @ (A @ V0)
    ref = np.linalg.eigvalsh(0.5 * (H + H.T))
    norm = np.abs(ref).max()
    # off-diagonal rest 1e-14 |H|_F, plus the rounding of 10 sweeps of n rotations each
    assert np.abs(theta - ref).max() <= 1e-13 * max(1.0, np.sqrt(ns) / 4) * norm
    assert np.abs(V.T @ V - np.eye(ns)).max() <= 1e-13
    # the Ritz vectors diagonalise H inside the span: ||V^T A V - diag|| <= 1e-13 sqrt(n) ||H||
    T = V.T @ (A @ V)
    assert np.linalg.norm(T - np.diag(theta)) <= 1e-13 * np.sqrt(ns) * np.linalg.norm(ref)
    R = A @ V - V * theta
    assert np.abs(np.linalg.norm(R, axis=0) - resid).max() <= 1e-12 * norm


@pytest.mark.parametrize("ns", [2, 14, 16, 18, 32, 34, 96, 130, 260])
def test_orders(ns):
    _check(fd_inputs.random_symmetric_csr(601, 9, ns), ns, ns)


@pytest.mark.parametrize("ns", [16, 34, 48, 96])
def test_eigenvectors_are_final(ns):
    """What the rotations leave off the diagonal is rounding, in every one of 24 problems.
    About u |H| in each of the n^2 entries is n u |H|, sqrt(n) u of the Ritz values' norm
    (which n values of that size have): four times that."""
    for seed in range(24):
        csr = fd_inputs.random_symmetric_csr(600, 9, seed)
        A = mat.to_scipy(csr)
        V0 = np.linalg.qr(fd_inputs.random_block(600, ns, seed))[0]
        theta, _, V = _ritz(csr, V0)
        T = V.T @ (A @ V)
        off = np.linalg.norm(T - np.diag(np.diag(T))) / np.linalg.norm(theta)
        assert off <= 4 * np.sqrt(ns) * 2.0 ** -53, seed


@pytest.mark.parametrize("scale", [1e-290, 1e-20, 1e150])
def test_scales(scale):
    p, c, v = fd_inputs.random_symmetric_csr(301, 9, 3)
    V0 = np.linalg.qr(fd_inputs.random_block(301, 24, 5))[0]
    A = mat.to_scipy((p, c, v))
    theta, _, _ = _ritz((p, c, v * scale), V0)
    ref = np.linalg.eigvalsh(V0.T @ (A @ V0))
    assert np.abs(theta / scale - ref).max() <= 1e-13 * np.abs(ref).max()


@pytest.mark.parametrize("gap", [0.0, 1e-13, 1e-9])
def test_clusters(gap):
    # eigenvalues in clusters of 8, `gap` apart within a cluster: H has them all
    D = ns = 48
    lam = np.repeat(np.arange(6) - 2.0, 8) + gap * np.tile(np.arange(8), 6)
    Q = np.linalg.qr(fd_inputs.random_block(D, D, 1))[0]
    H = Q @ np.diag(lam) @ Q.T
    H = 0.5 * (H + H.T)
    ptr = np.arange(0, D * D + 1, D, dtype=np.int64)
    csr = (ptr, np.tile(np.arange(D, dtype=np.int32), D), H.reshape(-1).copy())
    _check(csr, ns, 2)


@pytest.mark.parametrize("tiny", [1e-320, 1e-300, 1e-45, 1e-40, 1e-36, 1e-31, 1e-20])
def test_tiny_couplings_of_equal_diagonal_entries(tiny):
    # V = the first 16 unit vectors: H is the leading block of the matrix
    D = 40
    H = np.eye(D)
    H[0, 9] = H[9, 0] = H[2, 3] = H[3, 2] = tiny
    ptr = np.arange(0, D * D + 1, D, dtype=np.int64)
    csr = (ptr, np.tile(np.arange(D, dtype=np.int32), D), H.reshape(-1).copy())
    theta, resid, V = _ritz(csr, np.eye(D)[:, :16].copy())
    assert np.abs(theta - 1.0).max() <= 1e-15 and np.abs(V.T @ V - np.eye(16)).max() <= 1e-14
    assert resid.max() <= 1e-15


def test_nan_gives_nan():
    p, c, v = fd_inputs.random_symmetric_csr(120, 5, 3)
    V0 = np.linalg.qr(fd_inputs.random_block(120, 20, 5))[0]
    v = v.copy()
    v[0] = np.nan
    theta, _, _ = _ritz((p, c, v), V0)
    assert np.all(np.isnan(theta))
