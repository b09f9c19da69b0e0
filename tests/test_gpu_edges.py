"""GPU parity of single kernels at the sizes where their tiles, splits and dispatch rules
change: tile edges and remainders, the smallest sizes, both sides of every rule."""
import numpy as np
import pytest

import synth
from oracle import scloop, sox as osox
from gpu_common import check, pkg_built, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = torch_cuda()
    pkg = pkg_built()
    hs = {p: pkg.Handle(p) for p in ("fp64", "f16x2")}
    yield torch, pkg, hs
    for h in hs.values():
        h.close()


@pytest.mark.parametrize("n,N", [(1, 5), (7, 64), (8, 65), (9, 127), (16, 128), (17, 129), (33, 66), (64, 130),
                                 (65, 257)])
def test_mixed_tensor_and_half_transform_tiles(env, n, N):
    """Split-precision bare SOX where the mixed tensor's 8 x 16 column tiles, its 64 / 128 row
    tiles and the half transform's 128-column tiles end inside, on and past an edge."""
    torch, pkg, hs = env
    w = synth.molecule(300 + n, n, N, 4, 100.0, 1)
    p = pkg.problem(n, N, 4, 1, w.beta)
    G, X, V = to_dev(torch, w.G, w.X, w.V)
    S = torch.full_like(G, float("nan"))
    pkg.sox_sigma(hs["f16x2"], p, G, X, V, S)
    pkg.sox_check_device(hs["f16x2"])
    check(S.cpu().numpy(), osox.sox_sigma(w.X, w.V, w.G).real, "f16x2", f"n={n} N={N}", n=n, N=N)


@pytest.mark.parametrize("n,n_spin", [(1, 1), (2, 2), (31, 1), (33, 2), (110, 1), (111, 1)])
def test_dyson_and_mu_on_both_sides_of_the_shared_memory_rule(env, n, n_spin):
    """Systems inverted in shared memory (n <= 110) and through the augmented elimination:
    G(i w) against numpy's inverse with a condition-scaled bound, mu against the oracle's bisection."""
    torch, pkg, hs = env
    h = hs["fp64"]
    rng = np.random.default_rng(n)
    n_tau, beta, n_max, mu0 = 5, 4.0, 6 if n > 40 else 40, 0.1
    F = rng.standard_normal((n_spin, n, n)) / np.sqrt(n)
    F = 0.5 * (F + np.swapaxes(F, 1, 2))
    om = scloop.fermionic_frequencies(beta, n_max)
    S_tau = 0.05 * rng.standard_normal((n_spin, n_tau, n, n)) / np.sqrt(n)
    S_iw = 0.05 * (rng.standard_normal((n_spin, om.size, n, n)) + 1j * rng.standard_normal((n_spin, om.size, n, n)))
    S_iw /= np.sqrt(n)
    p = pkg.problem(n, 8, n_tau, n_spin, beta)
    Fd, Swd, Std, omd = to_dev(torch, F, S_iw, S_tau, om)
    out = torch.empty(n_spin, om.size, n, n, dtype=torch.complex128, device="cuda")
    pkg.sox_dyson(h, p, omd, mu0, Fd, Swd, out)
    for s in range(n_spin):
        ref = scloop.dyson(om, mu0, F[s], S_iw[s])
        A = (1j * om + mu0)[:, None, None] * np.eye(n) - F[s] - S_iw[s]
        # the forward error of an inverse with partial pivoting: n eps cond(A), a factor 8 to spare
        bound = 8 * n * 2.0 ** -53 * np.linalg.cond(A).max() * np.abs(ref).max()
        assert np.abs(out[s].cpu().numpy() - ref).max() <= bound
    target = 0.5 * n * n_spin
    got = pkg.sox_find_mu(h, p, omd, target, Fd, Swd, Std)
    ref_mu = scloop.find_mu(om, beta, target, list(F), list(S_iw), list(S_tau))
    assert abs(got - ref_mu) < 1e-9


def test_find_mu_limits(env):
    """max_iter ends the bisection early (the midpoint after that many halvings), and a
    singular system is reported."""
    torch, pkg, hs = env
    h = hs["fp64"]
    n, beta = 3, 4.0
    om = scloop.fermionic_frequencies(beta, 8)
    F = np.diag([-0.5, 0.1, 0.7])[None]
    p = pkg.problem(n, 4, 3, 1, beta)
    Fd, omd = to_dev(torch, F, om)
    zt, zw = np.zeros((3, n, n)), np.zeros((om.size, n, n), complex)
    for it in (1, 2, 7):
        got = pkg.sox_find_mu(h, p, omd, 1.5, Fd, lo=-8.0, hi=8.0, max_iter=it)
        ref = scloop.find_mu(om, beta, 1.5, [F[0]], [zw], [zt], lo=-8.0, hi=8.0, iters=it)
        assert abs(got - ref) < 1e-12
    zero, = to_dev(torch, np.zeros(2))
    with pytest.raises(pkg.SoxError):
        pkg.sox_find_mu(h, p, zero, 1.5, to_dev(torch, np.zeros((1, n, n)))[0], lo=-1.0, hi=1.0)


def _exact_projections(X, G):
    """X G, (X G^T), X G X^T in extended precision (rounded to FP64 only at the end)."""
    Xl, Gl = X.astype(np.longdouble), G.astype(np.longdouble)
    gr = np.stack([Xl @ g for g in Gl])
    gw = np.stack([g @ Xl.T for g in Gl])
    return gr, gw, np.stack([r @ Xl.T for r in gr])


# (n, N, batches): K = n at the ends of a 16-wide step, a 32-wide chunk, a 128-wide window
# (the 2^-55 and 2^-52 forms of the sums); rows at the ends of the 128 x 64 tiles; the last
# two stay on the FP64 pipe
@pytest.mark.parametrize("n,N,nb", [(15, 129, 600), (16, 64, 1000), (17, 128, 500), (33, 127, 120), (64, 65, 64),
                                    (127, 130, 10), (128, 128, 10), (129, 191, 6), (260, 70, 6), (5, 40, 4), (1, 7, 2)])
def test_fp64_products_from_digit_slices(env, n, N, nb):
    """thc_project_G against extended precision.  Bound per element: K terms whose factors are
    rounded at 2^-56 of twice the row maximum (2^-54 a term together), the final rounding and the
    dropped digit products below one more unit: (K + 4) 2^-53 of the maxima's product."""
    torch, pkg, hs = env
    rng = np.random.default_rng(1000 * n + N)
    G = rng.standard_normal((1, 1, nb, n, n)) * np.exp2(rng.integers(-40, 40, size=(1, 1, nb, 1, 1)).astype(float))
    X = rng.standard_normal((1, N, n))
    p = pkg.problem(n, N, nb, 1, 10.0)
    Gd, Xd = to_dev(torch, G, X)
    out = [torch.full(s, float("nan"), dtype=torch.float64, device="cuda")
           for s in ((1, 1, nb, N, n), (1, 1, nb, n, N), (1, 1, nb, N, N))]
    pkg.thc_project_G(hs["fp64"], p, Gd, Xd, *out)
    pkg.sox_check_device(hs["fp64"])
    ref = _exact_projections(X[0], G[0, 0])
    eps = (n + 4) * 2.0 ** -53
    gmax = np.abs(G[0, 0]).max(axis=(1, 2))[:, None, None]
    xmax = np.abs(X).max()
    got = [o.cpu().numpy()[0, 0] for o in out]
    assert (np.abs(got[0] - ref[0]) <= eps * xmax * gmax).all()
    assert (np.abs(got[1] - ref[1]) <= eps * xmax * gmax).all()
    # the second product's factor G_Rq carries the first one's error: K more times its bound
    rmax = np.abs(ref[0]).max(axis=(1, 2))[:, None, None].astype(float)
    assert (np.abs(got[2] - ref[2]) <= eps * xmax * rmax + n * xmax * eps * xmax * gmax).all()
    # not further from the exact product than FP64 arithmetic is
    f64 = np.stack([X[0] @ g for g in G[0, 0]])
    err = lambda a: float(np.sqrt((((a - ref[0]) / gmax) ** 2).sum()))  # noqa: E731
    assert err(got[0]) <= 1.5 * err(f64) + n * 2.0 ** -54


def test_fp64_products_with_zeros_infinities_and_nans(env):
    """Zero rows, subnormals, infinities and NaNs through the sliced product as through FP64."""
    torch, pkg, hs = env
    n, N, nb = 24, 96, 400
    rng = np.random.default_rng(3)
    G, X = rng.standard_normal((1, 1, nb, n, n)), rng.standard_normal((1, N, n))
    X[0, 5] = 0.0
    G[0, 0, 1] = 0.0
    G[0, 0, 2] *= 1e-310
    G[0, 0, 3, 2, 7] = np.inf
    G[0, 0, 4, 2, 7], G[0, 0, 4, 9, 7] = np.inf, -np.inf
    G[0, 0, 5, 0, 0] = np.nan
    G[0, 0, 6] *= 1e300
    p = pkg.problem(n, N, nb, 1, 10.0)
    Gd, Xd = to_dev(torch, G, X)
    gr = torch.zeros(1, 1, nb, N, n, dtype=torch.float64, device="cuda")
    pkg.thc_project_G(hs["fp64"], p, Gd, Xd, gr)
    got = gr.cpu().numpy()[0, 0]
    with np.errstate(all="ignore"):
        ref = np.stack([np.einsum("Ru,uq->Rq", X[0], g) for g in G[0, 0]])
    assert (np.isnan(got) == np.isnan(ref)).all()
    assert (np.isinf(got) == np.isinf(ref)).all() and (np.sign(got[np.isinf(ref)]) == np.sign(ref[np.isinf(ref)])).all()
    fin = np.isfinite(ref)
    cmax = np.where(np.isfinite(G[0, 0]), np.abs(G[0, 0]), 0.0).max(axis=1)[:, None, :]
    bound = (n + 4) * 2.0 ** -52 * np.abs(X).max() * np.broadcast_to(cmax, ref.shape) + 1e-320
    assert (np.abs(got - np.where(fin, ref, 0.0))[fin] <= bound[fin]).all()
    assert (got[:, 5][np.isfinite(G[0, 0]).all(axis=(1, 2))] == 0.0).all() and (got[1] == 0.0).all()


# n on both sides of a 16-wide step, a 32-wide chunk and the 128-wide window; N at the ends of
# the 128 x 32 tiles; the first two shapes stay on the FP64 pipe
@pytest.mark.parametrize("n,N,n_tau,v", [(3, 9, 4, None), (9, 64, 2, None), (16, 128, 6, None), (17, 129, 5, (3, 11)),
                                         (33, 160, 4, None), (64, 96, 3, None), (128, 33, 4, None), (130, 161, 2, None)])
def test_fp64_chain_from_digit_slices(env, n, N, n_tau, v):
    torch, pkg, hs = env
    w = synth.molecule(500 + n, n, N, n_tau, 30.0, 1)
    p = pkg.problem(n, N, n_tau, 1, w.beta)
    G, X, V = to_dev(torch, w.G, w.X, w.V)
    S = torch.full_like(G, float("nan"))
    with pkg.Handle("fp64") as h:
        if v:   # the two parts of a partition add up to the whole
            S1 = torch.empty_like(G)
            pkg.sox_set_v_range(h, 0, v[0])
            pkg.sox_sigma(h, p, G, X, V, S)
            for a, b in ((v[0], v[1]), (v[1], n)):
                pkg.sox_set_v_range(h, a, b)
                pkg.sox_sigma(h, p, G, X, V, S1)
                S += S1
        else:
            pkg.sox_sigma(h, p, G, X, V, S)
        pkg.sox_check_device(h)
    check(S.cpu().numpy(), osox.sox_sigma(w.X, w.V, w.G).real, "fp64", f"n={n} N={N}")


# N on both sides of the blocked solve's rule (64), of a 32-column block, of the 8-column inner
# blocks of a single large system; the larger ones leave shared memory for part of the way
@pytest.mark.parametrize("N", [1, 8, 63, 64, 65, 95, 130, 301, 1100])
def test_w_static_blocks_and_pivots(env, N):
    """W = (1 - V Pi)^-1 V with a V that forces row exchanges, against numpy's LU: the
    forward error bound of a solve with partial pivoting, N eps cond times a factor 8."""
    torch, pkg, hs = env
    rng = np.random.default_rng(N)
    V = rng.standard_normal((N, N)) / np.sqrt(N)
    Pi = rng.standard_normal((N, N)) / np.sqrt(N)
    K = np.eye(N) - V @ Pi
    p = pkg.problem(2, N, 2, 1, 10.0)
    Vd, Pd = to_dev(torch, V, Pi)
    W = torch.full((N, N), float("nan"), dtype=torch.float64, device="cuda")
    pkg.sox_w_static(hs["fp64"], p, Vd, Pd, W)
    pkg.sox_check_device(hs["fp64"])
    ref = np.linalg.solve(K, V)
    bound = 8 * N * 2.0 ** -53 * np.linalg.cond(K) * np.abs(ref).max()
    assert np.abs(W.cpu().numpy() - ref).max() <= bound


@pytest.mark.parametrize("N", [40, 96])
def test_w_static_reports_a_singular_system(env, N):
    torch, pkg, hs = env
    V, Pi = np.eye(N), np.eye(N)
    Pi[3, 3] = 0.5   # 1 - V Pi = diag(0, 0, 0, 1/2, 0, ...)
    p = pkg.problem(2, N, 2, 1, 10.0)
    Vd, Pd = to_dev(torch, V, Pi)
    with pytest.raises(pkg.SoxError):
        pkg.sox_w_static(hs["fp64"], p, Vd, Pd, torch.empty_like(Vd))


@pytest.mark.parametrize("nk,n,N,n_tau,M", [((2, 1, 1), 3, 70, 5, 2), ((1, 2, 2), 5, 97, 12, 4), ((3, 1, 1), 17, 130, 9, 3)])
def test_w_dynamic_of_solids_through_slices(env, nk, n, N, n_tau, M):
    """Complex products and the blocked complex solve at ragged sizes against the oracle."""
    from oracle import kpoints

    torch, pkg, hs = env
    w = synth.solid(40 + n, nk, n, N, n_tau, 20.0)
    _, Tf, _ = synth.bosonic_transforms(w.tau, w.beta, M)
    p = pkg.problem(n, N, n_tau, 1, w.beta, nk=nk, dtype=1)
    G, X, V, F = to_dev(torch, *(np.asarray(a, dtype=complex) for a in (w.G, w.X, w.V, Tf)))
    out = torch.full((w.n_k, 2 * M + 1, N, N), complex(float("nan"), 0.0), dtype=torch.complex128, device="cuda")
    pkg.sox_w_dynamic(hs["fp64"], p, G, X, V, F, 2 * M + 1, out)
    pkg.sox_check_device(hs["fp64"])
    ref = kpoints.w_dynamic(w.V, kpoints.pi_omega(w.X, w.G[0], Tf, nk))
    assert np.abs(out.cpu().numpy() - ref).max() <= 1e-10 * np.abs(ref).max()


def _random_dynamic(rng, n, N, n_tau, M, nk=None):
    """Inputs of the dynamic calls with random transforms and screening (any n_tau)."""
    w = synth.solid(70 + n, nk, n, N, n_tau, 10.0) if nk else synth.molecule(70 + n, n, N, n_tau, 10.0)
    Tf, Ti = (0.3 * (rng.standard_normal(s) + 1j * rng.standard_normal(s)) for s in ((M, n_tau), (n_tau, M)))
    shape = (w.X.shape[0], M, N, N) if nk else (M, N, N)
    Wd = rng.standard_normal(shape) / N   # real for molecules
    if nk:
        Wd = Wd + 1j * rng.standard_normal(shape) / N
    return w, Tf, Ti, Wd


def _dynamic(env, w, Tf, Ti, Wd, nk=None, scale=1.0):
    torch, pkg, hs = env
    h = hs["f16x2"]
    p = pkg.problem(w.n, w.N, w.n_tau, 1, w.beta, **(dict(nk=nk, dtype=1) if nk else {}))
    cast = complex if nk else float
    G, X, V = to_dev(torch, *(np.asarray(a, dtype=cast) for a in (w.G * scale, w.X, w.V)))
    F, I, W = to_dev(torch, Tf, Ti, Wd)
    S = torch.full_like(G, float("nan"))
    pkg.sosex_dynamic_sigma(h, p, G, X, V, W, F, I, Tf.shape[0], S)
    pkg.sox_check_device(h)
    return S.cpu().numpy()


@pytest.mark.parametrize("n,N,n_tau,M", [(1, 5, 2, 1), (7, 33, 3, 2), (8, 128, 4, 3), (9, 129, 2, 65), (33, 64, 65, 2)])
def test_dynamic_splits_and_maxima(env, n, N, n_tau, M):
    """FP16 pairs from integers and tensor maxima from the products' own tiles: N n off the 128
    columns of a tile, one row, K at 64 and 65, and a propagator 2^20 times smaller
    (every scale is a power of two: the same pairs, so the same bound on Sigma / 2^-60)."""
    from oracle import dynamic

    rng = np.random.default_rng(n)
    w, Tf, Ti, Wd = _random_dynamic(rng, n, N, n_tau, M)
    ref = dynamic.sosex_dynamic_sigma(w.X, w.V, Wd, Tf, Ti, w.G).real
    bar = 2e-6 * np.abs(ref).max()   # 22-bit pairs, FP32 sums
    for scale in (1.0, 2.0 ** -20):
        got = _dynamic(env, w, Tf, Ti, Wd, scale=scale) / scale ** 3
        assert np.abs(got - ref).max() <= bar, scale


@pytest.mark.parametrize("nk,n,N,n_tau,M", [((2, 1, 1), 3, 5, 2, 1), ((1, 2, 1), 2, 7, 4, 2), ((1, 1, 3), 5, 12, 5, 3),
                                            ((2, 1, 1), 3, 33, 9, 2), ((1, 1, 2), 4, 31, 129, 3)])
def test_solid_dynamic_pairs_of_the_time_products(env, nk, n, N, n_tau, M):
    """One, two, four and 32 lanes per row, times that fill no whole chunk of four, and more times
    than the lanes of a row keep; pair rows whose pitch is no multiple of 64 values."""
    from oracle import kpoints

    rng = np.random.default_rng(n_tau)
    w, Tf, Ti, Wd = _random_dynamic(rng, n, N, n_tau, M, nk)
    ref = kpoints.sosex_dynamic_sigma(w.X, w.V, Wd, Tf, Ti, w.G, nk)
    got = _dynamic(env, w, Tf, Ti, Wd, nk=nk)
    assert np.abs(got - ref).max() <= 2e-6 * np.abs(ref).max()


@pytest.mark.parametrize("nk,n,N,n_tau,M", [((1, 1, 2), 4, 16, 32, 16), ((1, 1, 2), 5, 13, 32, 16),
                                            ((1, 1, 2), 5, 13, 33, 17), ((2, 1, 1), 3, 50, 8, 7)])
def test_solid_transforms_with_exchanged_roles(env, nk, n, N, n_tau, M):
    """Transforms of 32 and 33 rows, 128 and 130 columns (both sides of the rule that puts the
    columns on the tile's rows), and K = 16 and 17 of the register and the shared-tile split."""
    from oracle import kpoints

    rng = np.random.default_rng(100 + n_tau)
    w, Tf, Ti, Wd = _random_dynamic(rng, n, N, n_tau, M, nk)
    ref = kpoints.sosex_dynamic_sigma(w.X, w.V, Wd, Tf, Ti, w.G, nk)
    got = _dynamic(env, w, Tf, Ti, Wd, nk=nk)
    assert np.abs(got - ref).max() <= 2e-6 * np.abs(ref).max()


@pytest.mark.parametrize("nk", [(4, 1, 1), (1, 5, 1), (1, 3, 4), (2, 1, 3)])
def test_w_dynamic_mesh_sides(env, nk):
    """Mesh transforms by butterflies (sides of 2, 3, 4) and by the twiddle matrix, along every axis."""
    from oracle import kpoints

    torch, pkg, hs = env
    n, N, n_tau, M = 3, 11, 6, 2
    w = synth.solid(90, nk, n, N, n_tau, 20.0)
    _, Tf, _ = synth.bosonic_transforms(w.tau, w.beta, M)
    p = pkg.problem(n, N, n_tau, 1, w.beta, nk=nk, dtype=1)
    G, X, V, F = to_dev(torch, *(np.asarray(a, dtype=complex) for a in (w.G, w.X, w.V, Tf)))
    out = torch.full((w.n_k, 2 * M + 1, N, N), complex(float("nan"), 0.0), dtype=torch.complex128, device="cuda")
    pkg.sox_w_dynamic(hs["fp64"], p, G, X, V, F, 2 * M + 1, out)
    pkg.sox_check_device(hs["fp64"])
    ref = kpoints.w_dynamic(w.V, kpoints.pi_omega(w.X, w.G[0], Tf, nk))
    assert np.abs(out.cpu().numpy() - ref).max() <= 1e-10 * np.abs(ref).max()


@pytest.mark.parametrize("n,N", [(32, 127), (33, 128), (46, 129)])
def test_split_adjoint_windows_of_k(env, n, N):
    """K = n^2 of one window (1024), one and a little, two and a little: the products of the
    adjoint's end in one launch that adds the windows in registers."""
    from oracle import grid, phi
    from test_gpu_phi import _grads_with

    torch, pkg, hs = env
    w = synth.molecule(120 + n, n, N, 3, 3.0)
    wt = grid.clenshaw_curtis(w.n_tau, w.beta)
    gX, gV = _grads_with(torch, pkg, hs["f16x2"], w, wt, [1.0])
    _, _, rX, rV = phi.phi_and_grads(w.X[0], w.V[0], w.G[0, 0], wt)
    assert np.abs(gX - rX).max() <= 2e-5 * np.abs(rX).max()
    assert np.abs(gV - rV).max() <= 2e-5 * np.abs(rV).max()
