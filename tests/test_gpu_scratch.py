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
