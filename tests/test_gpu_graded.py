"""FP64 entry points on data whose rows, columns or systems span many orders of magnitude:
accuracy relative to the sum of the magnitudes of an element's terms, not to the largest entries."""
import numpy as np
import pytest

import synth
from oracle import sox as osox
from gpu_common import pkg_built, to_dev, torch_cuda

pytestmark = pytest.mark.gpu
LD = np.longdouble


@pytest.fixture(scope="module")
def env():
    torch, pkg = torch_cuda(), pkg_built()
    h = pkg.Handle("fp64")
    yield torch, pkg, h
    h.close()


def _eliminate(A, N, dtype):
    """A column at a time with partial pivoting on [K | V]; the right half."""
    A = A.astype(dtype)
    for k in range(N):
        p = k + int(np.argmax(np.abs(A[k:, k])))
        A[[k, p]] = A[[p, k]]
        A[k, k:] = A[k, k:] * (dtype(1) / A[k, k])
        f = A[:, k].copy()
        f[k] = 0
        A[:, k + 1:] -= np.outer(f, A[k, k + 1:])
    return A[:, N:]


def _row_error(W, ref):
    return float((np.abs(W - ref).max(axis=1) / np.abs(ref).max(axis=1)).max())


# blocks of 32 and a rest, on one SM and across the device
@pytest.mark.parametrize("N", [64, 96, 130, 200])
@pytest.mark.parametrize("kind", ["large", "graded"])
def test_w_static_as_accurate_as_the_elimination_by_columns(env, N, kind):
    """V = Z Z^T 1e6 (cond(1 - V Pi) about 1e5 to 1e7, blocks of the matrix worse than it), and D V, Pi
    D^-1 with D of 2^-20 to 2^20.  Per row of W, relative to the extended-precision elimination of
    the same K: no more than 8 times (graded: 256 times, cond(D K D^-1) being 1e19) the error of the
    elimination by columns in FP64.  A block's explicit inverse is off by 60 to 4e5 times."""
    torch, pkg, h = env
    rng = np.random.default_rng(N)
    Z = rng.standard_normal((N, N))
    Z /= np.linalg.norm(Z, axis=0) * (1 + np.arange(N))
    Y = rng.standard_normal((N, N))
    V, Pi = Z @ Z.T, -(Y @ Y.T) / N / 10
    if kind == "large":
        V = V * 1e6
    else:
        d = np.exp2(rng.integers(-20, 21, N).astype(float))
        V, Pi = d[:, None] * V, Pi / d[None, :]
    K = np.eye(N) - V @ Pi
    Kl = np.eye(N, dtype=LD) - V.astype(LD) @ Pi.astype(LD)
    ref = _eliminate(np.hstack([Kl, V.astype(LD)]), N, LD)
    by_columns = _row_error(_eliminate(np.hstack([K, V]), N, np.float64), ref)
    p = pkg.problem(2, N, 2, 1, 10.0)
    Vd, Pd = to_dev(torch, V, Pi)
    W = torch.full((N, N), float("nan"), dtype=torch.float64, device="cuda")
    pkg.sox_w_static(h, p, Vd, Pd, W)
    pkg.sox_check_device(h)
    assert _row_error(W.cpu().numpy(), ref) <= (8 if kind == "large" else 256) * by_columns


@pytest.mark.parametrize("N", [96, 130])
def test_w_static_of_subnormal_values(env, N):
    """V of 1e-309 with Pi of 1e308: every product of the solve's right half leaves the normal range and
    is summed again from its sources.  The forward error of a solve, on values with a spacing of 2^-1074."""
    torch, pkg, h = env
    rng = np.random.default_rng(N)
    Z = rng.standard_normal((N, N)) / np.sqrt(N)
    Y = rng.standard_normal((N, N)) / np.sqrt(N)
    V, Pi = (Z @ Z.T) * 1e-309, -(Y @ Y.T) * 0.5e308
    K = np.eye(N) - V.astype(LD) @ Pi.astype(LD)
    ref = _eliminate(np.hstack([K, V.astype(LD)]), N, LD)
    p = pkg.problem(2, N, 2, 1, 10.0)
    Vd, Pd = to_dev(torch, V, Pi)
    W = torch.full((N, N), float("nan"), dtype=torch.float64, device="cuda")
    pkg.sox_w_static(h, p, Vd, Pd, W)
    pkg.sox_check_device(h)
    bound = 8 * N * np.linalg.cond(K.astype(float)) * (2.0 ** -53 * np.abs(ref).max() + LD(2.0) ** -1074)
    assert (np.abs(W.cpu().numpy() - ref) <= bound).all()


@pytest.mark.parametrize("nk,n,N", [((2, 1, 1), 5, 97), ((1, 1, 3), 4, 130)])
def test_w_dynamic_of_a_graded_basis(env, nk, n, N):
    """Rows of X times D and V between D^-2 and D^-2, D powers of two: the bubble has two factors of X per
    index, so W is D^-2 W D^-2, to the bound of the ungraded call (1e-10 of the largest)."""
    torch, pkg, h = env
    rng = np.random.default_rng(N)
    w = synth.solid(140, nk, n, N, 6, 20.0)
    _, Tf, _ = synth.bosonic_transforms(w.tau, w.beta, 2)
    p = pkg.problem(n, N, w.n_tau, 1, w.beta, nk=nk, dtype=1)
    d = np.exp2(rng.integers(-4, 5, N).astype(float))
    dd = (d[:, None] * d[None, :]) ** 2
    res = []
    for X, V in ((w.X, w.V), (w.X * d[:, None], w.V / dd)):
        Gd, Xd, Vd, F = to_dev(torch, *(np.asarray(a, dtype=complex) for a in (w.G, X, V, Tf)))
        out = torch.full((w.n_k, 5, N, N), complex(float("nan"), 0.0), dtype=torch.complex128, device="cuda")
        pkg.sox_w_dynamic(h, p, Gd, Xd, Vd, F, 5, out)
        pkg.sox_check_device(h)
        res.append(out.cpu().numpy())
    got = res[1] * dd
    assert np.abs(got - res[0]).max() <= 1e-10 * np.abs(res[0]).max()


def _digits(K):
    """A digit product is good to (1.1 K + 9) 2^-54 of the product of the maxima, and an element whose
    terms' magnitudes do not sum to 2^-6 of it is not taken from one: its error by that sum."""
    return (1.1 * K + 9) * 2.0 ** -48


@pytest.mark.parametrize("n,N,nb", [(2, 130, 3000), (33, 127, 120), (64, 65, 64), (130, 129, 6)])
@pytest.mark.parametrize("form", ["rows", "both", "diagonal"])
def test_projections_of_graded_rows(env, n, N, nb, form):
    """Rows of X that fall off over 200 powers of two, against G that is dense, falls off the other way
    or is diagonal: every element to the bound of a digit product by the sum of its terms' magnitudes
    (G_PQ: of two products)."""
    torch, pkg, h = env
    rng = np.random.default_rng(n + N)
    G, X = rng.standard_normal((nb, n, n)), rng.standard_normal((N, n))
    X *= np.exp2(-rng.integers(0, 200, size=(N, n)).astype(float))
    if form == "both":
        f = np.exp2(-100.0 * np.arange(n) / max(n - 1, 1))
        X = rng.standard_normal((N, n)) * f
        G = G * f[::-1, None]
    if form == "diagonal":
        G = np.eye(n) * rng.standard_normal((nb, 1, n))
    p = pkg.problem(n, N, nb, 1, 10.0)
    Gd, Xd = to_dev(torch, G[None, None], X[None])
    out = [torch.full(s, float("nan"), dtype=torch.float64, device="cuda")
           for s in ((1, 1, nb, N, n), (1, 1, nb, n, N), (1, 1, nb, N, N))]
    pkg.thc_project_G(h, p, Gd, Xd, *out)
    pkg.sox_check_device(h)
    for b in {0, nb // 2, nb - 1}:
        g, x = G[b].astype(LD), X.astype(LD)
        gr, gw, gq = (o[0, 0, b].cpu().numpy() for o in out)
        ag, ax = np.abs(g), np.abs(x)
        assert (np.abs(gr - x @ g) <= _digits(n) * (ax @ ag) + 1e-320).all()
        assert (np.abs(gw - g @ x.T) <= _digits(n) * (ag @ ax.T) + 1e-320).all()
        assert (np.abs(gq - x @ g @ x.T) <= 2.1 * _digits(n) * (ax @ ag @ ax.T) + 1e-320).all()


def test_fp64_sigma_of_graded_orbitals(env):
    """Orbital columns of X over 2^60 and G between the inverse factors: Sigma (r, t) carries the columns'
    factors, and keeps its digits in the smallest of them (five chained products of at most N
    terms, each to its bound by the magnitudes)."""
    torch, pkg, h = env
    n, N, T = 33, 160, 4
    w = synth.molecule(150, n, N, T, 10.0)
    f = np.exp2(np.round(np.linspace(0, 60, n)))
    X, G = w.X / f, w.G * (f[:, None] * f[None, :])
    p = pkg.problem(n, N, T, 1, w.beta)
    Gd, Xd, Vd = to_dev(torch, G, X, w.V)
    S = torch.full_like(Gd, float("nan"))
    pkg.sox_sigma(h, p, Gd, Xd, Vd, S)
    pkg.sox_check_device(h)
    ref = osox.sox_sigma(w.X, w.V, w.G).real
    mag = np.abs(osox.sox_sigma(np.abs(w.X), np.abs(w.V), np.abs(w.G)).real)
    got = S.cpu().numpy() * (f[:, None] * f[None, :])
    assert (np.abs(got - ref) <= 5 * _digits(N) * mag).all()


@pytest.mark.parametrize("N", [40, 64])
def test_w_dynamic_reports_a_system_whose_pivots_underflow(env, N):
    """The last pivot of 1 - V Pi is 1e-200: the square of its modulus is no number to divide by, and the
    call says so (below and above the rule of the block solve)."""
    torch, pkg, h = env
    G = np.zeros((1, 1, 2, N, N), complex)
    G[..., range(N), range(N)] = 0.5
    p, q = N - 2, N - 1   # Pi = G(0) o G(1)^T: 1 on the diagonal, 1e-200 and 1/4 beside it
    G[..., p, p] = G[..., q, q] = 1.0
    G[0, 0, 0, p, q] = G[0, 0, 1, q, p] = 1e-100
    G[0, 0, 0, q, p] = G[0, 0, 1, p, q] = 0.5
    p = pkg.problem(N, N, 2, 1, 10.0, nk=(1, 1, 1), dtype=1)
    Gd, Xd, Vd, F = to_dev(torch, G, np.eye(N, dtype=complex)[None], np.eye(N, dtype=complex)[None],
                           np.array([[-1.0 + 0j, 0.0]]))
    out = torch.empty(1, 1, N, N, dtype=torch.complex128, device="cuda")
    with pytest.raises(pkg.SoxError) as e:
        pkg.sox_w_dynamic(h, p, Gd, Xd, Vd, F, 1, out)
    assert e.value.code == 1
