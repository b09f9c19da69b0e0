"""Scratch memory of the FP64 products: where it lies, how it is sized, and what the handle's
workspace limit makes of it."""
import numpy as np
import pytest

import synth
from oracle import grid
from gpu_common import pkg_built, to_dev, torch_cuda
from test_gpu_phi import _grads_with

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    return torch_cuda(), pkg_built()


@pytest.mark.parametrize("n,N,n_tau,n_spin", [(20, 80, 600, 1), (8, 40, 3200, 2)])
def test_adjoint_of_a_long_grid_in_chunks_of_one_time(env, n, N, n_tau, n_spin):
    """The digits of the FP64 projections of all times are larger than the buffers of a chunk of one:
    they may not lie on them.  Same gradients as in one chunk up to the split path's bound
    (2e-5 of the largest, for either of the two)."""
    torch, pkg = env
    w = synth.molecule(130 + n, n, N, n_tau, 20.0, n_spin=n_spin)
    wt = grid.clenshaw_curtis(n_tau, w.beta)
    dphi = [1.0, -0.5][:n_spin]
    with pkg.Handle("f16x2") as h:
        rX, rV = _grads_with(torch, pkg, h, w, wt, dphi)
    with pkg.Handle("f16x2", workspace_limit=1) as h:
        gX, gV = _grads_with(torch, pkg, h, w, wt, dphi)
    assert np.abs(gX - rX).max() <= 4e-5 * np.abs(rX).max()
    assert np.abs(gV - rV).max() <= 4e-5 * np.abs(rV).max()


def _w_dynamic(torch, pkg, h, w, Tf, nk):
    p = pkg.problem(w.n, w.N, w.n_tau, 1, w.beta, nk=nk, dtype=1)
    G, X, V, F = to_dev(torch, *(np.asarray(a, dtype=complex) for a in (w.G, w.X, w.V, Tf)))
    out = torch.full((w.n_k, len(Tf), w.N, w.N), complex(float("nan"), 0.0), dtype=torch.complex128, device="cuda")
    pkg.sox_w_dynamic(h, p, G, X, V, F, len(Tf), out)
    pkg.sox_check_device(h)
    return out


@pytest.mark.parametrize("nk,N,n_omega", [((3, 3, 3), 300, 25), ((4, 4, 4), 200, 21)])
def test_w_dynamic_on_a_handle_made_for_it(env, nk, N, n_omega):
    """Only half of the +-Omega systems are solved: the scratch that is reserved for all of them has
    to hold the passes of half of them too.  One frequency against a call of its own."""
    torch, pkg = env
    w = synth.solid(131, nk, 3, N, 4, 20.0)
    _, Tf, _ = synth.bosonic_transforms(w.tau, w.beta, (n_omega - 1) // 2)
    with pkg.Handle("fp64") as h:
        out = _w_dynamic(torch, pkg, h, w, Tf, nk)
    with pkg.Handle("fp64") as h:
        one = _w_dynamic(torch, pkg, h, w, Tf[2:3], nk)
    assert float((out[:, 2] - one[:, 0]).abs().max()) <= 1e-10 * float(one.abs().max())


def _free(torch):
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_digits_of_a_product_stay_within_the_limit(env):
    """G_Rq, G_wP and G_PQ of 1024 times: the digits of the last product's operands take 0.5 GB at once,
    passes of 64 MB with that limit, and the same numbers either way."""
    torch, pkg = env
    n, N, T = 64, 512, 1024
    rng = np.random.default_rng(5)
    p = pkg.problem(n, N, T, 1, 10.0)
    G, X = to_dev(torch, rng.standard_normal((1, 1, T, n, n)), rng.standard_normal((1, N, n)))
    outs, used = [], []
    for limit in (0, 64 << 20):
        out = [torch.full(s, float("nan"), dtype=torch.float64, device="cuda")
               for s in ((1, 1, T, N, n), (1, 1, T, n, N), (1, 1, T, N, N))]
        with pkg.Handle("fp64", workspace_limit=limit) as h:
            before = _free(torch)
            pkg.thc_project_G(h, p, G, X, *out)
            used.append(before - _free(torch))
            pkg.sox_check_device(h)
        outs.append(out)
    assert all(bool((a == b).all()) for a, b in zip(*outs))
    assert used[0] >= 400 << 20 and used[1] <= 160 << 20   # two operands of a pass


@pytest.mark.parametrize("case", ["solve", "columns"])
def test_passes_of_the_solve_give_the_same_numbers(env, case):
    """One system (or 1024 columns) per pass against all at once."""
    torch, pkg = env
    res = []
    if case == "solve":
        w = synth.solid(132, (2, 2, 1), 3, 70, 4, 20.0)
        _, Tf, _ = synth.bosonic_transforms(w.tau, w.beta, 3)
        for limit in (0, 1):
            with pkg.Handle("fp64", workspace_limit=limit) as h:
                res.append(_w_dynamic(torch, pkg, h, w, Tf, w.nk))
    else:
        N, rng = 1100, np.random.default_rng(6)
        V, Pi = to_dev(torch, *(rng.standard_normal((N, N)) / np.sqrt(N) for _ in range(2)))
        for limit in (0, 1):
            with pkg.Handle("fp64", workspace_limit=limit) as h:
                res.append(torch.empty_like(V))
                pkg.sox_w_static(h, pkg.problem(2, N, 2, 1, 10.0), V, Pi, res[-1])
                pkg.sox_check_device(h)
    assert bool((res[0] == res[1]).all())


@pytest.mark.parametrize("n_t", [1, 8, 37])
def test_iw_to_tau_in_blocks_of_times(env, n_t):
    """8192 frequencies and 4096 times would be 0.5 GB of phases: 64 MB are taken.  In blocks of eight times
    (the smallest limit) the numbers are those of one block."""
    torch, pkg = env
    n, n_w, rng = 3, 8192, np.random.default_rng(7)
    om = (2 * np.arange(-n_w // 2, n_w // 2) + 1) * np.pi / 5.0
    tau = np.sort(rng.uniform(0, 5.0, 4096))
    G = rng.standard_normal((2, n_w, n, n)) + 1j * rng.standard_normal((2, n_w, n, n))
    Gd, tails, omd, td = to_dev(torch, G, rng.standard_normal((2, 3, n, n)), om, tau)
    p = pkg.problem(n, 4, 8, 2, 5.0)
    with pkg.Handle("fp64") as h:
        before = _free(torch)
        out = torch.empty(2, 4096, n, n, dtype=torch.float64, device="cuda")
        pkg.sox_iw_to_tau(h, p, omd, Gd, tails, td, out)
        assert before - _free(torch) <= 80 << 20
        few = torch.empty(2, n_t, n, n, dtype=torch.float64, device="cuda")
        pkg.sox_iw_to_tau(h, p, omd, Gd, tails, td[:n_t].contiguous(), few)
    with pkg.Handle("fp64", workspace_limit=1) as h:
        one = torch.empty_like(few)
        pkg.sox_iw_to_tau(h, p, omd, Gd, tails, td[:n_t].contiguous(), one)
        pkg.sox_check_device(h)
    assert bool((few == out[:, :n_t]).all()) and bool((one == few).all())


def test_static_solid_takes_the_memory_there_is(env):
    """A chunk of all 30 times would take 1.9 GB, one time 0.2 GB: with 1 GB left on the device the call
    runs, in smaller chunks and to the same numbers."""
    torch, pkg = env
    w = synth.solid(133, (2, 2, 1), 26, 300, 30, 100.0)
    p = pkg.problem(w.n, w.N, w.n_tau, 1, w.beta, nk=w.nk, dtype=1)
    G, X, V = to_dev(torch, w.G, w.X, w.V)
    S = [torch.full_like(G, complex("nan")) for _ in range(2)]
    with pkg.Handle("f16x2") as h:
        pkg.sox_sigma(h, p, G, X, V, S[0])
        pkg.sox_check_device(h)
    torch.cuda.empty_cache()
    fill = torch.empty(_free(torch) - (1 << 30), dtype=torch.uint8, device="cuda")
    try:
        with pkg.Handle("f16x2") as h:
            pkg.sox_sigma(h, p, G, X, V, S[1])
            pkg.sox_check_device(h)
    finally:
        del fill
        torch.cuda.empty_cache()
    assert bool((S[0] == S[1]).all())
