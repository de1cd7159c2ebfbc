"""Filters of every degree from 2 to 9: the accumulator takes three terms every
third step and the rest at the last one, so each remainder is a case of its own."""
import numpy as np
import pytest

import fd_inputs
from gpu_util import U32, U64, filter_tolerance
from oracle import chebyshev as ch
from oracle import lanczos
from oracle import matrices as mat

pytestmark = pytest.mark.gpu

MATRICES = [
    ("anderson3d:L=11,W=3,seed=5", 32, 1),
    ("chain:n=777,t=1", 64, 8),                                             # permuted rows
    ("hubbard:n_sites=7,n_up=3,n_dn=4,t=1,U=4,bc=periodic,kron=1", 32, 1),  # matrix-free
]


@pytest.mark.parametrize("spec,C,sigma", MATRICES)
@pytest.mark.parametrize("prec", ["f64", "f32", "ff"])
@pytest.mark.parametrize("n", range(2, 10))
def test_accumulation_remainders(spec, C, sigma, prec, n):
    import torch

    import paper_2209_01974_gb300 as fd
    nb = 8
    ctx = fd.fd_create(0)
    csr = mat.build(spec.replace(",kron=1", ""))
    A = fd.fd_build_matrix(ctx, spec, C=C, sigma=sigma)
    V0 = fd_inputs.random_block(len(csr[0]) - 1, nb, n).astype(np.float32).astype(np.float64)
    lo, hi = lanczos.gershgorin(csr)
    alpha, beta = ch.scale_params(lo - 0.01, hi + 0.01)
    mu = np.random.default_rng(n).uniform(0.5, 1.0, n + 1) * (-1.0) ** np.arange(n + 1)
    out = torch.from_numpy(V0).cuda()
    W = torch.empty_like(out)
    if prec != "f64":
        V = torch.empty(V0.shape + ((2,) if prec == "ff" else ()), dtype=torch.float32, device="cuda")
        W = torch.empty_like(V)
        fd.fd_copy_block(ctx, out, V)
        fd.fd_filter(ctx, A, V, mu, alpha, beta, W, torch.empty_like(V))
        fd.fd_copy_block(ctx, V, out)
    else:
        fd.fd_filter(ctx, A, out, mu, alpha, beta, W, torch.empty_like(W))
    ref = ch.cheb_filter(mat.to_scipy(csr), V0, mu, alpha, beta)
    u = {"f64": U64, "f32": U32, "ff": 2.0 ** -45}[prec]
    assert np.all(np.abs(out.cpu().numpy() - ref) <= filter_tolerance(csr, mu, alpha, beta, V0, u))


def _random_ragged(D, seed):
    return fd_inputs.random_symmetric_csr(D, 9, seed, max_row=40)


# rows around the splits of the one-launch filter (clusters of 1, 2, 4, 8 CTAs, rows
# in fours) and, from 40,000 on, the launched steps
@pytest.mark.parametrize("D", [3, 31, 33, 130, 1023, 1500, 4999, 40001])
@pytest.mark.parametrize("nb,prec", [(2, "f64"), (4, "f32"), (8, "ff"), (16, "f64"), (32, "f32"), (64, "f64"),
                                     (64, "ff"), (128, "f32")])
@pytest.mark.parametrize("sigma", [1, 64])
def test_sizes(D, nb, prec, sigma):
    import torch

    import paper_2209_01974_gb300 as fd
    ctx = fd.fd_create(0)
    csr = _random_ragged(D, D + nb)
    A = fd.fd_matrix_from_csr(ctx, *csr, C=32, sigma=sigma)
    n = 7
    V0 = fd_inputs.random_block(D, nb, n).astype(np.float32).astype(np.float64)
    lo, hi = lanczos.gershgorin(csr)
    alpha, beta = ch.scale_params(lo - 0.01, hi + 0.01)
    mu = np.random.default_rng(n).uniform(0.5, 1.0, n + 1)
    ld = 2 * nb                                   # a bundle of a wider block
    big = torch.zeros((D, ld), dtype=torch.float64, device="cuda")
    big[:, nb:] = torch.from_numpy(V0)
    shape, dtype = ((D, nb), torch.float64) if prec == "f64" else ((D, nb), torch.float32)
    if prec == "ff":
        shape = (D, nb, 2)
    W1, W2 = (torch.empty(shape, dtype=dtype, device="cuda") for _ in range(2))
    if prec == "f64":
        fd.fd_filter(ctx, A, big[:, nb:], mu, alpha, beta, W1, W2)
    else:
        V = torch.empty(shape, dtype=dtype, device="cuda")
        fd.fd_copy_block(ctx, big[:, nb:], V)
        fd.fd_filter(ctx, A, V, mu, alpha, beta, W1, W2)
        fd.fd_copy_block(ctx, V, big[:, nb:])
    out = big.cpu().numpy()
    assert np.all(out[:, :nb] == 0.0)
    ref = ch.cheb_filter(mat.to_scipy(csr), V0, mu, alpha, beta)
    # two roundings more per row: the scaled entries and the scaled diagonal
    u = {"f64": U64, "f32": U32, "ff": 2.0 ** -45}[prec]
    assert np.all(np.abs(out[:, nb:] - ref) <= filter_tolerance(csr, mu, alpha, beta, V0, u))


@pytest.mark.parametrize("n", [998, 999, 1000, 1001, 2500])
@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_steps_split_over_launches(n, prec):
    """The one-launch filter takes at most 999 steps at a time."""
    import torch

    import paper_2209_01974_gb300 as fd
    ctx = fd.fd_create(0)
    spec = "anderson3d:L=7,W=3,seed=5"
    csr = mat.build(spec)
    A = fd.fd_build_matrix(ctx, spec)
    lo, hi = lanczos.gershgorin(csr)
    alpha, beta = ch.scale_params(lo - 0.01, hi + 0.01)
    mu = ch.filter_coeffs(0.1, 0.15, n)
    V0 = fd_inputs.random_block(343, 8, n).astype(np.float32).astype(np.float64)
    dtype = torch.float64 if prec == "f64" else torch.float32
    V = torch.from_numpy(V0).to(dtype).cuda()
    fd.fd_filter(ctx, A, V, mu, alpha, beta, torch.empty_like(V), torch.empty_like(V))
    ref = ch.cheb_filter(mat.to_scipy(csr), V0, mu, alpha, beta)
    # the errors of the steps add up like sqrt(n) (their signs vary); 40 sqrt(n) u |ref|
    u = U64 if prec == "f64" else U32
    assert np.linalg.norm(V.cpu().numpy() - ref) <= 40 * np.sqrt(n) * u * np.linalg.norm(V0)


def _filter_case(fd, ctx, spec, n, dtype, seed, alpha=None):
    import torch
    A = fd.fd_build_matrix(ctx, spec)
    csr = mat.build(spec.replace(",kron=1", ""))
    lo, hi = lanczos.gershgorin(csr)
    alpha, beta = ch.scale_params(lo - 0.01, hi + 0.01)
    mu = np.random.default_rng(seed).uniform(0.5, 1.0, n + 1) / (n + 1)
    V0 = fd_inputs.random_block(len(csr[0]) - 1, 8, seed)
    V = torch.from_numpy(V0).cuda()
    ref = ch.cheb_filter(mat.to_scipy(csr), V0, mu, alpha, beta)
    return A, V, mu, alpha, beta, torch.empty_like(V), torch.empty_like(V), ref, \
        filter_tolerance(csr, mu, alpha, beta, V0, U64)


LARGE = "anderson3d:L=34,W=3,seed=5"     # 39,304 rows: launched steps


@pytest.mark.parametrize("spec", [LARGE, "hubbard:n_sites=7,n_up=3,n_dn=4,t=1,U=4,bc=periodic,kron=1"])
def test_scaled_matrix_refused_or_captured(spec):
    """A filter without its scaled-matrix buffer (workspace cap, stream capture)
    gives the same result to rounding."""
    import torch

    import paper_2209_01974_gb300 as fd
    ctx = fd.fd_create(0)
    A, V, mu, alpha, beta, W1, W2, ref, tol = _filter_case(fd, ctx, spec, 14, torch.float64, 3)
    V0 = V.clone()
    fd.fd_filter(ctx, A, V, mu, alpha, beta, W1, W2)
    assert np.all(np.abs(V.cpu().numpy() - ref) <= tol)
    ctx2 = fd.fd_create(0)
    fd.fd_set_workspace_limit(ctx2, 8)
    V.copy_(V0)
    fd.fd_filter(ctx2, A, V, mu, alpha, beta, W1, W2)
    assert np.all(np.abs(V.cpu().numpy() - ref) <= tol)
    g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        fd.fd_set_stream(ctx, s.cuda_stream)
        V.copy_(V0)
        with torch.cuda.graph(g, stream=s):
            fd.fd_filter(ctx, A, V, mu, alpha, beta, W1, W2)
        g.replay()
    torch.cuda.synchronize()
    assert np.all(np.abs(V.cpu().numpy() - ref) <= tol)


def test_filters_of_one_context_on_two_streams():
    """Two matrices and scalings through one context, its stream changed between
    the calls without waiting: the scaled-matrix buffer is not overwritten early."""
    import torch

    import paper_2209_01974_gb300 as fd
    ctx = fd.fd_create(0)
    a = _filter_case(fd, ctx, LARGE, 60, torch.float64, 1)
    b = _filter_case(fd, ctx, "anderson3d:L=33,W=9,seed=8", 60, torch.float64, 2)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    for (A, V, mu, alpha, beta, W1, W2, _, _), s in zip((a, b), streams):
        fd.fd_set_stream(ctx, s.cuda_stream)
        fd.fd_filter(ctx, A, V, mu, alpha, beta, W1, W2)
    torch.cuda.synchronize()
    for c in (a, b):
        assert np.all(np.abs(c[1].cpu().numpy() - c[7]) <= c[8])


@pytest.mark.parametrize("D,nb", [(30000, 8), (28000, 16), (30000, 32), (9000, 128)])
def test_float_float_long_rows(D, nb):
    """The float-float step's CTAs per SM by the length of rows and the size of the grid."""
    import torch

    import paper_2209_01974_gb300 as fd
    ctx = fd.fd_create(0)
    csr = fd_inputs.random_symmetric_csr(D, 17, nb, max_row=60)
    A = fd.fd_matrix_from_csr(ctx, *csr)
    assert A.info["nnz"] >= 12 * D
    V0 = fd_inputs.random_block(D, nb, 3).astype(np.float32).astype(np.float64)
    lo, hi = lanczos.gershgorin(csr)
    alpha, beta = ch.scale_params(lo - 0.01, hi + 0.01)
    mu = np.random.default_rng(1).uniform(0.5, 1.0, 14)
    out = torch.from_numpy(V0).cuda()
    V = torch.empty((D, nb, 2), dtype=torch.float32, device="cuda")
    fd.fd_copy_block(ctx, out, V)
    fd.fd_filter(ctx, A, V, mu, alpha, beta, torch.empty_like(V), torch.empty_like(V))
    fd.fd_copy_block(ctx, V, out)
    ref = ch.cheb_filter(mat.to_scipy(csr), V0, mu, alpha, beta)
    assert np.all(np.abs(out.cpu().numpy() - ref) <= filter_tolerance(csr, mu, alpha, beta, V0, 2.0 ** -45))


def test_scaled_matrix_across_destroyed_streams():
    """The scaled matrix of one filter is not overwritten by the next one's while steps on
    a stream that has since been destroyed still read it; the new stream may get the old
    one's handle."""
    import ctypes

    import torch

    import paper_2209_01974_gb300 as fd
    rt = torch.cuda.cudart()
    ctx = fd.fd_create(0)
    specs = ["anderson3d:L=60,W=3,seed=5", "anderson3d:L=60,W=3,seed=6"]
    mats = [fd.fd_build_matrix(ctx, s) for s in specs]
    D, nb = 60 ** 3, 16
    mu = np.random.default_rng(3).uniform(0.5, 1.0, 101)
    V0 = torch.randn((D, nb), dtype=torch.float64, device="cuda")

    def run(stream_of, sync):
        out = []
        for A in mats:
            V, W1, W2 = V0.clone(), torch.empty_like(V0), torch.empty_like(V0)
            torch.cuda.synchronize() if sync else torch.cuda.current_stream().synchronize()
            s = stream_of()
            fd.fd_set_stream(ctx, s.value)
            fd.fd_filter(ctx, A, V, mu, 0.12, 0.01, W1, W2)
            fd.fd_set_stream(ctx, None)
            assert int(rt.cudaStreamDestroy(s.value)) == 0   # returns at once, the work goes on
            out.append((V, W1, W2))
        torch.cuda.synchronize()
        return [o[0] for o in out]

    def fresh():
        s = ctypes.c_void_p()
        assert int(rt.cudaStreamCreate(ctypes.addressof(s))) == 0
        return s
    apart, close = run(fresh, True), run(fresh, False)
    assert all(torch.equal(a, b) for a, b in zip(apart, close))
