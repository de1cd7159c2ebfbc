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
