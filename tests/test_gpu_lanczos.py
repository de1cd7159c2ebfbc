"""Inclusion intervals from the one-launch Lanczos kernel against the oracle:
few rows, more steps than rows, an invariant start (early stop), permuted rows,
sizes around the rows of a CTA."""
import numpy as np
import pytest

from oracle import lanczos
from oracle import matrices as mat

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("spec,C,sigma", [
    ("chain:n=2,t=1", 32, 1), ("chain:n=3,t=1", 32, 1), ("chain:n=63,t=1", 32, 1), ("chain:n=65,t=1", 32, 1),
    ("anderson3d:L=11,W=3,seed=5", 64, 1), ("chain:n=777,t=1", 96, 8), ("anderson3d:L=24,W=16,seed=2", 32, 1),
])
@pytest.mark.parametrize("steps", [1, 2, 20, 50])
def test_bounds_match_oracle(spec, C, sigma, steps):
    import paper_2209_01974_gb300 as fd
    ctx = fd.fd_create(0)
    csr = mat.build(spec)
    A = fd.fd_build_matrix(ctx, spec, C=C, sigma=sigma)
    lo, hi = fd.fd_spectral_bounds(ctx, A, steps, 7)
    olo, ohi = lanczos.inclusion_interval(csr, steps, 7)
    # extreme Ritz values are well conditioned; the residual bound beta |s| loses
    # digits only where it is itself far below the interval's width
    assert max(abs(lo - olo), abs(hi - ohi)) <= 1e-9 * (ohi - olo)


@pytest.mark.parametrize("spec,steps", [("chain:n=155649,t=1", 9), ("anderson3d:L=56,W=5,seed=1", 20),
                                        ("chain:n=500003,t=1", 17), ("anderson3d:L=90,W=5,seed=2", 20)])
def test_many_rows_match_oracle(spec, steps):
    """Two to four CTAs per SM, with one to three tiles of vectors."""
    import paper_2209_01974_gb300 as fd
    ctx = fd.fd_create(0)
    csr = mat.build(spec)
    lo, hi = fd.fd_spectral_bounds(ctx, fd.fd_build_matrix(ctx, spec), steps, 3)
    olo, ohi = lanczos.inclusion_interval(csr, steps, 3)
    assert max(abs(lo - olo), abs(hi - ohi)) <= 1e-9 * (ohi - olo)


def test_more_steps_than_the_default_shared_memory_holds():
    """A solve may ask for thousands of steps: 6,200 coefficients are 48.4 KB.  (Two
    eigenvalues, so that the recurrence itself ends after two steps.)"""
    import paper_2209_01974_gb300 as fd
    ctx = fd.fd_create(0)

    def solve(D, steps):
        csr = (np.arange(D + 1, dtype=np.int64), np.arange(D, dtype=np.int32), np.where(np.arange(D) % 3, 2.0, -1.0))
        A = fd.fd_matrix_from_csr(ctx, *csr)
        return fd.fd_solve(ctx, A, 1.9, 2.1, 1, 8, 10, 1e-9, raise_noconv=False, max_outer=1, lanczos_steps=steps)[2]
    for D in (7000, 200000):    # one and two CTAs per SM
        res = solve(D, 6200)
        assert np.allclose((res["lam_l"], res["lam_r"]), (-1.0, 2.0), rtol=0, atol=1e-12)
    with pytest.raises(fd.FDError) as e:
        solve(40000, 40000)
    assert e.value.status == fd.FD_ERR_ARG


def test_early_stop_on_an_invariant_subspace():
    import paper_2209_01974_gb300 as fd
    ctx = fd.fd_create(0)
    D = 500
    d = np.where(np.arange(D) % 3 == 0, -1.0, 2.0)   # two eigenvalues: two steps span everything
    csr = (np.arange(D + 1, dtype=np.int64), np.arange(D, dtype=np.int32), d)
    A = fd.fd_matrix_from_csr(ctx, *csr)
    assert np.allclose(fd.fd_spectral_bounds(ctx, A, 20, 1), (-1.0, 2.0), rtol=0, atol=1e-12)
