"""Measured workloads of the filter-diagonalization library.

Every case is one call sequence that a program using the library makes, through
the public binding, at a size from the repository's configurations or a generic
one:

  filter       the Chebyshev filter phase of one outer FD iteration: every
               nb-wide bundle of the FP64 search block is converted to the sweep
               type, filtered, and put back (Alg. 2)
  ortho        Cholesky-QR of the search block
  ritz         the Rayleigh-Ritz step: Ritz values, vectors and residuals
  prepare      what precedes a solve with learned parameters: the inclusion
               interval (Lanczos) and the kernel-polynomial moments
  solve        a whole FD solve of one problem
  batch        a whole batched solve of several uneven problems

Inputs are made from the seed alone: Anderson and road-graph matrices take it
as their disorder seed, search blocks are normal-like.  exact() restates the
same quantities in plain NumPy / torch FP64.
"""
import math

import numpy as np
import torch

import paper_2209_01974_gb300 as fd

L2_BYTES = 126e6   # blocks larger than this cannot stay on the chip between degree steps
PRECS = ("f64", "f32", "ff")


# --------------------------------------------------------------------------- the cases
def listed():
    return [
        # config 1 (8-site Hubbard chain, 20 pairs): the smallest filters, 4,900
        # rows; launches and latency count
        dict(name="filter f64 hubbard8", path="filter", matrix="hubbard", size=8, nb=16, bundles=5,
             degree=100, prec="f64", C=32, sigma=1),
        # the benchmark's sweep: FP32 on the 2.1M-row stencil, far larger than L2
        dict(name="filter f32 stencil128", path="filter", matrix="anderson", size=128, nb=64, bundles=1,
             degree=40, prec="f32", C=32, sigma=1),
        # the default (FP64) sweep on the mid-size time-to-solution problem
        dict(name="filter f64 anderson48", path="filter", matrix="anderson", size=48, nb=32, bundles=4,
             degree=100, prec="f64", C=32, sigma=1),
        # the float-float finishing sweep on the same problem
        dict(name="filter ff anderson48", path="filter", matrix="anderson", size=48, nb=32, bundles=4,
             degree=100, prec="ff", C=32, sigma=1),
        # the wide many-body pattern: the 14-site ring (11.8M rows), matrix-free
        dict(name="filter f32 ring14", path="filter", matrix="ring", size=14, nb=32, bundles=1,
             degree=12, prec="f32", C=32, sigma=1),
        # ragged short rows (road-like graph Laplacian, odd side), FP32
        dict(name="filter f32 road1201", path="filter", matrix="road", size=1201, nb=32, bundles=1,
             degree=40, prec="f32", C=32, sigma=1),
        # orthonormalisation of the mid-size problem's block (32 pairs)
        dict(name="ortho 110592x128", path="ortho", rows=110592, ns=128),
        # and of the benchmark's block (100 pairs, N_s = 384)
        dict(name="ortho 2097152x384", path="ortho", rows=2097152, ns=384),
        # the Rayleigh-Ritz step of the mid-size problem
        dict(name="ritz anderson48x128", path="ritz", size=48, ns=128),
        # interval and moments of a mid-size problem (16 vectors, 48 moments as the
        # predictor's features take them)
        dict(name="prepare anderson48", path="prepare", size=48, moments=48, vectors=16),
        # a whole small solve, FP64 throughout (the default form)
        dict(name="solve f64 anderson12", path="solve", size=12, targets=12, nb=16, degree=60, prec="f64"),
        # a batch of uneven small problems, FP32 sweeps and float-float finish
        dict(name="batch 12 anderson10-14", path="batch", instances=12, lo=10, hi=14, targets=8, nb=8,
             degree=100, prec="f32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges the listed ones stand for."""
    path = rng.choice(["filter", "filter", "filter", "filter", "ortho", "ritz", "prepare", "solve", "batch"])
    if path == "filter":
        matrix = rng.choice(["anderson", "anderson", "road", "hubbard", "ring"])
        prec = rng.choice(PRECS)
        nb = rng.choice([8, 16, 32, 64])
        size = {"anderson": lambda: _log_int(rng, 12, 112), "road": lambda: _log_int(rng, 60, 1200),
                "hubbard": lambda: rng.choice([6, 7, 8, 9, 10]), "ring": lambda: rng.choice([8, 9, 10, 11, 12, 13])}[matrix]()
        # wide FP64-accurate blocks on the largest matrices would cost more than the listed cases
        rows = _rows(matrix, size)
        while rows * nb > (6e7 if prec == "f32" else 2e7) and nb > 8:
            nb //= 2
        degree = max(4, min(_log_int(rng, 10, 200), int(3e9 / (rows * nb)) if prec == "f32" else int(1e9 / (rows * nb))))
        sigma = 1 if matrix == "ring" else rng.choice([1, 1, 128])
        return dict(path="filter", matrix=matrix, size=size, nb=nb, bundles=rng.choice([1, 2, 3]), degree=degree,
                    prec=prec, C=rng.choice([32, 32, 64]), sigma=sigma)
    if path == "ortho":
        ns = rng.choice([16, 24, 48, 80, 96, 128, 200, 256, 384])
        rows = _log_int(rng, 1500, 1.5e6) | 1
        return dict(path="ortho", rows=rows, ns=ns)
    if path == "ritz":
        return dict(path="ritz", size=_log_int(rng, 14, 72), ns=rng.choice([16, 48, 80, 128, 192, 256]))
    if path == "prepare":
        return dict(path="prepare", size=_log_int(rng, 14, 64), moments=rng.choice([17, 48, 64, 128]),
                    vectors=rng.choice([4, 8, 16, 32]))
    if path == "solve":
        targets = rng.choice([8, 12, 16])
        return dict(path="solve", size=rng.choice([9, 10, 11, 12, 13, 14]), targets=targets,
                    nb=rng.choice([8, 16, 32]), degree=rng.choice([40, 60, 80]), prec=rng.choice(PRECS))
    lo = rng.choice([9, 10, 11])
    return dict(path="batch", instances=rng.choice([3, 5, 8, 11]), lo=lo, hi=lo + rng.choice([1, 2, 3]),
                targets=8, nb=rng.choice([8, 16]), degree=rng.choice([60, 100]), prec=rng.choice(["f64", "f32"]))


# --------------------------------------------------------------------------- sizes
HUBBARD_U = 4.0
ANDERSON_W = 16.0   # the time-to-solution problem's disorder (filters, ritz, prepare)
SOLVE_W = 12.0      # below the localisation transition: level repulsion, eigenvectors well defined
SOLVE_HALF = 0.01   # half width of the solves' windows around 0
SOLVE_NS = 8        # search vectors per wanted pair


def _rows(matrix, size):
    if matrix == "anderson":
        return size ** 3
    if matrix == "road":
        return size * size
    return math.comb(size, size // 2) ** 2


def _nnz(matrix, size):
    if matrix == "anderson":
        return 7 * size ** 3
    if matrix == "road":
        return int(3.6 * size * size)
    bonds = size - 1 if matrix == "hubbard" else size
    up = size // 2
    # a bond can be hopped over when exactly one of its ends is occupied
    per_spin = bonds * 2 * math.comb(size - 2, up - 1)
    dim = math.comb(size, up)
    return dim * dim + 2 * per_spin * dim


def _spec(matrix, size, seed):
    if matrix == "anderson":
        return f"anderson3d:L={size},W={ANDERSON_W},seed={seed}"
    if matrix == "road":
        return f"roadgraph:side={size},q=0.3,seed={seed}"
    half = size // 2
    bc = "open" if matrix == "hubbard" else "periodic,kron=1"
    return f"hubbard:n_sites={size},n_up={half},n_dn={half},t=1,U={HUBBARD_U},bc={bc}"


def _interval(matrix, size):
    """Gershgorin-type inclusion interval of the spectrum (closed form)."""
    if matrix == "anderson":
        return -6.0 - ANDERSON_W / 2, 6.0 + ANDERSON_W / 2
    if matrix == "road":
        return 0.0, 8.0
    hops = 2.0 * (size if matrix == "ring" else size - 1)
    return -hops, hops + HUBBARD_U * (size // 2)


def _filter_window(matrix, size):
    """Window well inside the spectrum, as FD's interior targets are, and its scaled form."""
    lo, hi = _interval(matrix, size)
    alpha, beta = 2.0 / (hi - lo), -(hi + lo) / (hi - lo)
    c = lo + 0.47 * (hi - lo)
    w = 0.01 * (hi - lo)
    return alpha, beta, alpha * (c - w) + beta, alpha * (c + w) + beta


def _block(rows, cols, seed, dtype=torch.float64):
    g = torch.Generator(device="cuda").manual_seed(1000003 * (seed % 100000) + 17)
    return torch.randn((rows, cols), dtype=torch.float32, device="cuda", generator=g).to(dtype)


def _search_block(rows, cols, seed):
    """FP64 normal-like block whose entries use the whole FP64 significand."""
    V = _block(rows, cols, seed)
    return V.mul_(1.0 + 1e-7 * math.pi).add_(V * V, alpha=1e-9 / 3)


def _ortho_block(rows, ns, seed):
    """A block as the filter leaves it: columns mixed, singular values over three decades."""
    g = torch.Generator(device="cuda").manual_seed(seed % 100000 + 5)
    M = torch.randn((ns, ns), dtype=torch.float64, device="cuda", generator=g)
    Q = torch.linalg.qr(M)[0] * torch.logspace(0, -3, ns, dtype=torch.float64, device="cuda")[None, :]
    V = _block(rows, ns, seed, torch.float32) @ Q.float()
    return V.double().mul_(1.0 + 1e-7 * math.pi).add_(V, alpha=1e-9 / 3)


# --------------------------------------------------------------------------- prepare and run
def prepare(case, seed):
    ctx = fd.fd_create(0)
    s = dict(case=case, seed=seed, ctx=ctx)
    path = case["path"]
    if path == "filter":
        s["A"] = fd.fd_build_matrix(ctx, _spec(case["matrix"], case["size"], seed), C=case["C"], sigma=case["sigma"])
        rows, nb, ns = _rows(case["matrix"], case["size"]), case["nb"], case["nb"] * case["bundles"]
        s["alpha"], s["beta"], xl, xr = _filter_window(case["matrix"], case["size"])
        s["mu"] = fd.fd_filter_coeffs(xl, xr, case["degree"])
        s["V"] = _search_block(rows, ns, seed)
        s["out"] = torch.empty_like(s["V"])
        if case["prec"] == "f64":
            shape, dtype = (rows, nb), torch.float64
        elif case["prec"] == "f32":
            shape, dtype = (rows, nb), torch.float32
            s["Vw"] = torch.empty(shape, dtype=dtype, device="cuda")
        else:
            shape, dtype = (rows, nb, 2), torch.float32
            s["Vw"] = torch.empty(shape, dtype=dtype, device="cuda")
        s["W1"] = torch.empty(shape, dtype=dtype, device="cuda")
        s["W2"] = torch.empty(shape, dtype=dtype, device="cuda")
    elif path == "ortho":
        s["V"] = _ortho_block(case["rows"], case["ns"], seed)
        s["out"] = torch.empty_like(s["V"])
    elif path == "ritz":
        s["A"] = fd.fd_build_matrix(ctx, _spec("anderson", case["size"], seed))
        s["V"] = _search_block(case["size"] ** 3, case["ns"], seed)
        fd.fd_orthonormalize(ctx, s["V"])
        s["out"], s["AV"] = torch.empty_like(s["V"]), torch.empty_like(s["V"])
        s["probe"] = _block(1, case["size"] ** 3, seed + 1)
    elif path == "prepare":
        s["A"] = fd.fd_build_matrix(ctx, _spec("anderson", case["size"], seed))
    elif path == "solve":
        s["A"] = fd.fd_build_matrix(ctx, f"anderson3d:L={case['size']},W={SOLVE_W},seed={seed}")
        s["X"] = torch.empty((case["size"] ** 3, case["targets"]), dtype=torch.float64, device="cuda")
    else:
        s["A"] = [fd.fd_build_matrix(ctx, f"anderson3d:L={L},W={SOLVE_W},seed={seed + k}")
                  for k, L in enumerate(_batch_sizes(case))]
        s["problems"] = [(-SOLVE_HALF, SOLVE_HALF, case["targets"], seed + k) for k in range(case["instances"])]
    return s


def _batch_sizes(case):
    return [case["lo"] + k % (case["hi"] - case["lo"] + 1) for k in range(case["instances"])]


def _form(prec):
    """Options of the three precision forms; the FP32 form finishes in float-float."""
    return dict(precision="f32", finish="ff") if prec == "f32" else dict(precision=prec)


def run(s):
    case, ctx, path = s["case"], s["ctx"], s["case"]["path"]
    if path == "filter":
        nb, V, out = case["nb"], s["V"], s["out"]
        for j in range(0, V.shape[1], nb):
            if case["prec"] == "f64":   # in place on the bundle's columns of the block
                fd.fd_copy_block(ctx, V[:, j:j + nb], out[:, j:j + nb])
                fd.fd_filter(ctx, s["A"], out[:, j:j + nb], s["mu"], s["alpha"], s["beta"], s["W1"], s["W2"])
            else:
                fd.fd_copy_block(ctx, V[:, j:j + nb], s["Vw"])
                fd.fd_filter(ctx, s["A"], s["Vw"], s["mu"], s["alpha"], s["beta"], s["W1"], s["W2"])
                fd.fd_copy_block(ctx, s["Vw"], out[:, j:j + nb])
        return out
    if path == "ortho":
        fd.fd_copy_block(ctx, s["V"], s["out"])
        fd.fd_orthonormalize(ctx, s["out"])
        return s["out"]
    if path == "ritz":
        fd.fd_copy_block(ctx, s["V"], s["out"])
        theta, resid = fd.fd_rayleigh_ritz(ctx, s["A"], s["out"], s["AV"])
        return [theta, resid] + _signed(s["out"], s["AV"], s["probe"])
    if path == "prepare":
        lo, hi = fd.fd_spectral_bounds(ctx, s["A"], 20, s["seed"])
        mu = fd.fd_kpm_moments(ctx, s["A"], case["moments"], case["vectors"], s["seed"], 2.0 / (hi - lo),
                               -(hi + lo) / (hi - lo))
        return [np.array([lo, hi]), mu]
    if path == "solve":
        theta, _, _ = fd.fd_solve(ctx, s["A"], -SOLVE_HALF, SOLVE_HALF, case["targets"], case["nb"], case["degree"],
                                  1e-9, X=s["X"], raise_noconv=False, seed=s["seed"], ns=SOLVE_NS * case["targets"],
                                  lam_l=-6.0 - SOLVE_W / 2, lam_r=6.0 + SOLVE_W / 2, **_form(case["prec"]))
        return [theta, s["X"]]
    # the batched call takes its intervals from Lanczos: enough steps that they hold the spectrum's tails
    out, _ = fd.fd_solve_batched(ctx, s["A"], s["problems"], case["nb"], case["degree"], 1e-9, raise_noconv=False,
                                 ns=SOLVE_NS * case["targets"], lanczos_steps=50, **_form(case["prec"]))
    return np.concatenate([theta for theta, _ in out])


def _signed(V, AV, probe):
    """Ritz vectors are defined up to sign: the one with a positive component along a fixed vector."""
    sign = torch.sign(probe @ V)
    return [V * sign, AV * sign]


# --------------------------------------------------------------------------- work
def work(case):
    path = case["path"]
    if path == "filter":
        rows, nnz = _rows(case["matrix"], case["size"]), _nnz(case["matrix"], case["size"])
        S, cols, n = (4 if case["prec"] == "f32" else 8), case["nb"] * case["bundles"], case["degree"]
        mat = 0 if case["matrix"] == "ring" else nnz * (S + 4)
        total = 16.0 * rows * cols + mat   # the FP64 block read and written, the matrix read
        if 2.0 * rows * case["nb"] * S > L2_BYTES:
            # every step reads two recurrence vectors, writes one and reads the matrix
            total += n * (3.0 * rows * cols * S + mat * case["bundles"])
        return {"bytes": total, "flops": (2.0 * nnz + 6.0 * rows) * cols * n}
    if path == "ortho":
        D, n = case["rows"], case["ns"]
        return {"bytes": 16.0 * D * n, "flops": 2 * (2.0 * D * n * n)}  # two triangular Grams and solves
    if path == "ritz":
        D, n = case["size"] ** 3, case["ns"]
        return {"bytes": 24.0 * D * n + 84.0 * D, "flops": 3.0 * D * n * n + 28.0 * D * n + 9.0 * n ** 3}
    if path == "prepare":
        D = case["size"] ** 3
        return {"bytes": 84.0 * D + 8.0 * D * case["vectors"],
                "flops": case["moments"] / 2 * case["vectors"] * 20.0 * D + 20 * (14.0 + 80.0) * D}
    if path == "solve":
        D, ns = case["size"] ** 3, SOLVE_NS * case["targets"]
        sweeps = 5 * 4 * 3.14 / (0.3 * ns / D)     # about five filters of degree 4 pi / dtheta
        return {"bytes": 84.0 * D + 8.0 * D * case["targets"], "flops": 20.0 * D * ns * sweeps}
    flops = 0.0
    ns = SOLVE_NS * case["targets"]
    for L in _batch_sizes(case):
        flops += 20.0 * L ** 3 * ns * 5 * 4 * 3.14 / (0.3 * ns / L ** 3)
    return {"bytes": sum(84.0 * L ** 3 for L in _batch_sizes(case)), "flops": flops}


# --------------------------------------------------------------------------- tolerances
# about four times the error against exact() that the listed cases and 80 draws showed
# (filters 7e-16 .. 5e-15, 4.5e-7 and 2e-14; ortho 3e-13 with singular values over
# three decades; ritz 9e-13, most for close Ritz values; prepare 2e-14).  A solve
# stops at residual 1e-9, so its vectors are right to 1e-9 over the gap between
# neighbouring eigenvalues, and its eigenvalues to far less.
def tolerance(case):
    path = case["path"]
    if path == "filter":
        return {"rel": {"f64": 2e-14, "f32": 2e-6, "ff": 1e-13}[case["prec"]]}
    return {"rel": {"ortho": 2e-12, "ritz": 1e-11, "prepare": 1e-13, "solve": 1e-6, "batch": 1e-9}[path]}


# --------------------------------------------------------------------------- exact values
# the library's counter-based SplitMix64 streams (Steele, Lea, Flood 2014), from
# their definition: key = mix(seed ^ mix(stream)), x_i = mix(key + (i + 1) GAMMA)
def _mix(z):
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def _raw(seed, stream, i):
    with np.errstate(over="ignore"):
        key = _mix(np.uint64(seed) ^ _mix(np.uint64(stream)))
        return _mix(key + (np.asarray(i, dtype=np.uint64) + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15))


def _uniform(seed, stream, i):
    return (_raw(seed, stream, i) >> np.uint64(11)).astype(np.float64) * 2.0 ** -53


def _normal_like(seed, stream, e):
    s = np.zeros(len(e), dtype=np.uint64)
    for t in range(12):
        s += _raw(seed, stream, np.asarray(e, dtype=np.uint64) * np.uint64(12) + np.uint64(t)) >> np.uint64(11)
    return s.astype(np.float64) * 2.0 ** -53 - 6.0


def _csr(rows, cols, vals, D):
    """torch CSR (FP64, on the GPU) of the given entries."""
    order = np.lexsort((cols, rows))
    ptr = np.zeros(D + 1, dtype=np.int64)
    np.cumsum(np.bincount(rows, minlength=D), out=ptr[1:])
    t = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (ptr, cols[order], vals[order])]
    return torch.sparse_csr_tensor(*t, size=(D, D))


def _anderson(L, W, seed):
    D = L ** 3
    i = np.arange(D)
    x, y, z = i % L, i // L % L, i // (L * L)
    nbr = [i, (x + 1) % L + L * (y + L * z), (x - 1) % L + L * (y + L * z), x + L * ((y + 1) % L + L * z),
           x + L * ((y - 1) % L + L * z), x + L * (y + L * ((z + 1) % L)), x + L * (y + L * ((z - 1) % L))]
    vals = np.full((7, D), -1.0)
    vals[0] = W * (_uniform(seed, 1, i) - 0.5)
    return _csr(np.tile(i, 7), np.concatenate(nbr), vals.reshape(-1), D)


def _road(side, q, seed):
    N = side * side
    i = np.arange(N)
    x, y = i % side, i // side
    coin = _uniform(seed, 7, i)
    tree_left = (x > 0) & ((y == 0) | (coin < 0.5))
    tree_down = (y > 0) & ((x == 0) | (coin >= 0.5))
    left = tree_left | ((x > 0) & (_uniform(seed, 8, 2 * i) < q))
    down = tree_down | ((y > 0) & (_uniform(seed, 8, 2 * i + 1) < q))
    a, b = np.concatenate([i[left], i[down]]), np.concatenate([i[left] - 1, i[down] - side])
    deg = (np.bincount(a, minlength=N) + np.bincount(b, minlength=N)).astype(np.float64)
    off = np.full(2 * len(a), -1.0)
    return _csr(np.concatenate([i, a, b]), np.concatenate([i, b, a]), np.concatenate([deg, off]), N)


def _spin(n, periodic):
    """One spin species of the Hubbard chain: states (ascending bit strings) and hopping CSR, t = 1."""
    states = np.array([b for b in range(1 << n) if bin(b).count("1") == n // 2])
    rank = np.full(1 << n, -1)
    rank[states] = np.arange(len(states))
    rows, cols, vals = [], [], []
    for i, j in [(k, k + 1) for k in range(n - 1)] + ([(0, n - 1)] if periodic else []):
        can = ((states >> i) & 1) != ((states >> j) & 1)
        between = ((1 << j) - 1) ^ ((1 << (i + 1)) - 1)
        passed = np.array([bin(b).count("1") for b in (states[can] & between)])
        rows.append(np.nonzero(can)[0])
        cols.append(rank[states[can] ^ ((1 << i) | (1 << j))])
        vals.append(-1.0 + 2.0 * (passed % 2))
    return states, _csr(np.concatenate(rows), np.concatenate(cols), np.concatenate(vals), len(states))


def _operator(matrix, size, seed):
    """x -> H x on FP64 blocks."""
    if matrix in ("anderson", "road"):
        A = _anderson(size, ANDERSON_W, seed) if matrix == "anderson" else _road(size, 0.3, seed)
        return lambda x: A @ x
    states, H = _spin(size, matrix == "ring")
    d = len(states)
    pop = torch.tensor([bin(k).count("1") for k in range(1 << size)], dtype=torch.float64, device="cuda")
    st = torch.from_numpy(states).cuda()
    diag = HUBBARD_U * pop[st[:, None] & st[None, :]]

    def apply(x):
        m = x.shape[1]
        x3 = x.view(d, d, m)
        y = (H @ x3.reshape(d, d * m)).view(d, d, m)
        y += (H @ x3.transpose(0, 1).reshape(d, d * m)).view(d, d, m).transpose(0, 1)
        y += diag[:, :, None] * x3
        return y.reshape(d * d, m)
    return apply


def _coefficients(xl, xr, n):
    """Jackson-damped Chebyshev coefficients of a window, 1 at its centre."""
    tl, tr = math.acos(xl), math.acos(xr)
    k = np.arange(1, n + 1)
    c = np.concatenate([[(tl - tr) / math.pi], 2 * (np.sin(k * tl) - np.sin(k * tr)) / (k * math.pi)])
    N, k = n + 1, np.arange(n + 1)
    a = math.pi / (N + 1)
    mu = c * ((N - k + 1) * np.cos(a * k) + np.sin(a * k) / math.tan(a)) / (N + 1)
    return mu / np.sum(mu * np.cos(k * math.acos(0.5 * (xl + xr))))


def _cholqr(V):
    for _ in range(2):
        R = torch.linalg.cholesky(V.T @ V, upper=True)
        V = torch.linalg.solve_triangular(R, V, upper=True, left=False)
    return V


def _nearest(ev, X, k):
    """The k eigenpairs nearest 0, ascending, largest entry of each vector positive."""
    sel = torch.sort(torch.argsort(ev.abs(), stable=True)[:k])[0]
    if X is None:
        return ev[sel]
    X = X[:, sel]
    return ev[sel], X * torch.sign(torch.gather(X, 0, X.abs().argmax(0, keepdim=True)))


def exact(case, seed):
    path = case["path"]
    if path == "filter":
        rows, ns = _rows(case["matrix"], case["size"]), case["nb"] * case["bundles"]
        H = _operator(case["matrix"], case["size"], seed)
        alpha, beta, xl, xr = _filter_window(case["matrix"], case["size"])
        mu = _coefficients(xl, xr, case["degree"])
        x0 = _search_block(rows, ns, seed)
        x1 = H(x0).mul_(alpha).add_(x0, alpha=beta)
        out = mu[0] * x0 + mu[1] * x1
        for k in range(2, case["degree"] + 1):
            x2 = H(x1).mul_(2 * alpha).add_(x1, alpha=2 * beta).sub_(x0)
            out.add_(x2, alpha=mu[k])
            x0, x1 = x1, x2
        return out
    if path == "ortho":
        return _cholqr(_ortho_block(case["rows"], case["ns"], seed))
    if path == "ritz":
        A = _anderson(case["size"], ANDERSON_W, seed)
        V = _cholqr(_search_block(case["size"] ** 3, case["ns"], seed))
        theta, Q = torch.linalg.eigh(V.T @ (A @ V))
        V = V @ Q
        AV = A @ V
        probe = _block(1, case["size"] ** 3, seed + 1)
        return [theta, torch.linalg.vector_norm(AV - theta * V, dim=0)] + _signed(V, AV, probe)
    if path == "prepare":
        return _exact_prepare(case, seed)
    if path == "solve":
        ev, X = torch.linalg.eigh(_anderson(case["size"], SOLVE_W, seed).to_dense())
        return list(_nearest(ev, X, case["targets"]))
    parts = []
    for k, L in enumerate(_batch_sizes(case)):
        ev = torch.linalg.eigvalsh(_anderson(L, SOLVE_W, seed + k).to_dense())
        parts.append(_nearest(ev, None, case["targets"]))
    return torch.cat(parts)


def _exact_prepare(case, seed):
    A = _anderson(case["size"], ANDERSON_W, seed)
    D, m = A.shape[0], 20
    diag = ANDERSON_W * (_uniform(seed, 1, np.arange(D)) - 0.5)
    q = torch.from_numpy(_normal_like(seed, 3, np.arange(D))).cuda()
    q /= q.norm()
    Q, a, b = [], [], []
    for _ in range(m):
        Q.append(q)
        w = (A @ q[:, None])[:, 0]
        a.append(float(q @ w))
        P = torch.stack(Q, 1)
        for _ in range(2):
            w = w - P @ (P.T @ w)
        b.append(float(w.norm()))
        q = w / b[-1]
    T = np.diag(a) + np.diag(b[:-1], 1) + np.diag(b[:-1], -1)
    th, S = np.linalg.eigh(T)
    span = th[-1] - th[0]
    lo = max(th[0] - abs(b[-1] * S[-1, 0]) - 0.01 * span, diag.min() - 6.0)
    hi = min(th[-1] + abs(b[-1] * S[-1, -1]) + 0.01 * span, diag.max() + 6.0)
    alpha, beta = 2.0 / (hi - lo), -(hi + lo) / (hi - lo)
    R = case["vectors"]
    x0 = torch.from_numpy(_normal_like(seed, 4, np.arange(D * R)).reshape(D, R)).cuda()
    r, mu = x0, [float((x0 * x0).sum())]
    x1 = alpha * (A @ x0) + beta * x0
    for k in range(1, case["moments"]):
        mu.append(float((r * x1).sum()))
        x0, x1 = x1, 2.0 * (alpha * (A @ x1) + beta * x1) - x0
    return [np.array([lo, hi]), np.array(mu) / (R * D)]
