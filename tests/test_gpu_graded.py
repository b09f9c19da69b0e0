"""FP64 entry points on data whose rows, columns or systems span many orders of magnitude:
accuracy relative to the sum of the magnitudes of an element's terms, not to the largest entries."""
import numpy as np
import pytest

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
