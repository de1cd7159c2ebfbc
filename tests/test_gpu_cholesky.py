"""Cholesky and triangular inverse through Cholesky-QR: orders around the 8-row
panels and the grid, graded blocks; block copies at every width and alignment."""
import os
import subprocess
import sys

import numpy as np
import pytest

import fd_inputs
pytestmark = pytest.mark.gpu


def _qr(V0):
    import torch

    import paper_2209_01974_gb300 as fd
    ctx = fd.fd_create(0)
    V = torch.from_numpy(V0).cuda()
    R = torch.empty((V0.shape[1],) * 2, dtype=torch.float64, device="cuda")
    passes = fd.fd_orthonormalize(ctx, V, R)
    return V.cpu().numpy(), R.cpu().numpy(), passes


@pytest.mark.parametrize("ns", [1, 2, 7, 8, 9, 15, 16, 17, 63, 65, 127, 153, 161, 200, 305, 600])
@pytest.mark.parametrize("spread", [0, 6])
def test_orders(ns, spread):
    D = 2 * ns + 37
    V0 = fd_inputs.random_block(D, ns, ns) * np.logspace(0, -spread, ns)[None, :]
    Q, R, passes = _qr(V0)
    assert passes == 2
    assert np.abs(Q.T @ Q - np.eye(ns)).max() <= 1e-14 * max(1.0, ns / 100)
    assert np.all(np.tril(R, -1) == 0.0)
    # R against LAPACK's up to row signs, column by column: each column's size sets its scale
    ref = np.linalg.qr(V0, mode="r")
    ref *= np.sign(np.diag(ref))[:, None]
    scale = np.linalg.norm(V0, axis=0)
    assert np.all(np.abs(R - ref) <= 1e-12 * np.sqrt(ns) * scale[None, :])


@pytest.mark.parametrize("exponent", [-500, -333, -1, 0, 1, 400, 501])
@pytest.mark.parametrize("ns", [3, 24, 40])
def test_pivots_of_every_size(ns, exponent):
    """Pivots down to 2^-1000 and up to 2^1002, even and odd powers of two side by side:
    scaling columns by powers of two scales R's columns by them and leaves Q."""
    D = 3 * ns + 50
    V0 = fd_inputs.random_block(D, ns, ns)
    scale = np.ldexp(1.0, exponent + np.arange(ns) % 3 - 1)
    Q, R, passes = _qr(V0 * scale[None, :])
    Q1, R1, _ = _qr(V0)
    assert passes == 2
    assert np.abs(Q - Q1).max() <= 1e-13 and np.abs(Q.T @ Q - np.eye(ns)).max() <= 1e-14
    assert np.abs(R / scale[None, :] - R1).max() <= 1e-13 * np.abs(R1).max()


def test_orders_whose_shared_memory_is_just_above_the_default():
    """From 727 on the triangular inverse's shared memory, static and dynamic, exceeds
    the 48 KB that a launch gets unasked.  In a process of its own: the larger limit
    stays with a kernel once a wider block has asked for it."""
    code = """
import numpy as np, torch
import fd_inputs, paper_2209_01974_gb300 as fd
ctx = fd.fd_create(0)
for ns in (726, 727, 768, 769, 1024):
    V = torch.from_numpy(fd_inputs.random_block(ns + 37, ns, ns)).cuda()
    assert fd.fd_orthonormalize(ctx, V) == 2
    Q = V.cpu().numpy()
    assert np.abs(Q.T @ Q - np.eye(ns)).max() <= 1e-14 * ns / 100, ns
"""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]


@pytest.mark.parametrize("n", [1, 3, 4, 6, 255, 256, 257, 1030])
@pytest.mark.parametrize("pad,shift", [(0, 0), (2, 2), (3, 1), (4, 0)])
def test_copy_block_widths(n, pad, shift):
    """Type conversions at widths and alignments with and without wide accesses."""
    _copies(67, n, pad, shift)


@pytest.mark.parametrize("D,n", [(1, 1), (3, 5000), (50, 1021), (20011, 7), (9731, 130), (3000, 1025)])
def test_copy_block_splits(D, n):
    """One and four rows per thread, several thread blocks along a row."""
    _copies(D, n, 1, 0)


def _copies(D, n, pad, shift):
    import torch

    import paper_2209_01974_gb300 as fd
    ctx = fd.fd_create(0)
    src = torch.from_numpy(fd_inputs.random_block(D, n, n)).cuda()
    big = torch.zeros((D, n + pad + shift), dtype=torch.float64, device="cuda")
    v64 = big[:, shift:shift + n]
    fd.fd_copy_block(ctx, src, v64)
    assert torch.equal(v64, src) and int((big != 0).sum()) == D * n
    v32 = torch.zeros((D, n + pad + shift), dtype=torch.float32, device="cuda")[:, shift:shift + n]
    fd.fd_copy_block(ctx, v64, v32)
    assert torch.equal(v32, src.float())
    fd.fd_copy_block(ctx, v32, v64)
    assert torch.equal(v64, src.float().double())
    vff = torch.zeros((D, n + pad + shift, 2), dtype=torch.float32, device="cuda")[:, shift:shift + n]
    fd.fd_copy_block(ctx, src, vff)
    hi = src.float()
    assert torch.equal(vff[..., 0], hi) and torch.equal(vff[..., 1], (src - hi.double()).float())
    fd.fd_copy_block(ctx, vff, v64)
    assert torch.equal(v64, hi.double() + (src - hi.double()).float().double())


@pytest.mark.parametrize("n", [1, 4, 5, 256, 1030])
@pytest.mark.parametrize("so,do", [(0, 1), (1, 0), (1, 1)])
def test_copy_block_pairs_between_8_byte_boundaries(n, so, do):
    """Float-float blocks that start at an odd float."""
    import torch

    import paper_2209_01974_gb300 as fd
    ctx = fd.fd_create(0)
    D = 67

    def block(off):
        return torch.zeros(2 * D * n + 1, dtype=torch.float32, device="cuda")[off:off + 2 * D * n].view(D, n, 2)
    src = torch.from_numpy(fd_inputs.random_block(D, n, n)).cuda()
    a, b = block(so), block(do)
    assert a.data_ptr() % 8 == 4 * so and b.data_ptr() % 8 == 4 * do
    fd.fd_copy_block(ctx, src, a)
    hi = src.float()
    assert torch.equal(a[..., 0], hi) and torch.equal(a[..., 1], (src - hi.double()).float())
    fd.fd_copy_block(ctx, a, b)
    assert torch.equal(a, b)
    back = torch.empty_like(src)
    fd.fd_copy_block(ctx, b, back)
    assert torch.equal(back, b[..., 0].double() + b[..., 1].double())
