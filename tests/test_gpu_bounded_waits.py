"""Waits that run out: every warp of a tensor-core kernel leaves, the call's status is a timeout and the
context stays usable.  (With an iteration cap of 1 the lanes of an epilogue warp see the end of a wait,
or the abort flag of another warp, at different times.)"""
import numpy as np
import pytest

import synth
from oracle import grid, sox as osox
from gpu_common import check, pkg_built, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call,prec", [("sigma", "fp64"), ("project", "fp64"), ("backward", "f16x2"), ("batch", "f16x2")])
def test_waits_that_run_out_end_the_whole_warp(call, prec):
    torch, pkg = torch_cuda(), pkg_built()
    w = synth.molecule(160, 64, 256, 4, 100.0)
    p = pkg.problem(w.n, w.N, w.n_tau, 1, w.beta)
    G, X, V, wt = to_dev(torch, w.G, w.X, w.V, grid.clenshaw_curtis(w.n_tau, w.beta))
    S = torch.empty_like(G)

    def run(h):
        if call == "sigma":
            pkg.sox_sigma(h, p, G, X, V, S)
        elif call == "project":
            pkg.thc_project_G(h, p, G, X, *(torch.empty(s, dtype=torch.float64, device="cuda")
                                            for s in ((1, 1, 4, 256, 64), (1, 1, 4, 64, 256), (1, 1, 4, 256, 256))))
        elif call == "backward":
            pkg.phi_sox_backward(h, p, G, X, V, wt, torch.ones(1, dtype=torch.float64, device="cuda"), None,
                                 torch.empty_like(X), torch.empty_like(V))
        else:
            pkg.sox_sigma_batch(h, [p, p], [G, G], [X, X], [V, V], [S, torch.empty_like(G)])

    with pkg.Handle(prec, spin_limit=1) as h:
        for _ in range(4):
            run(h)
            with pytest.raises(pkg.SoxError) as e:
                pkg.sox_check_device(h)
            assert e.value.code == 6
    with pkg.Handle(prec) as h:
        run(h)
        pkg.sox_sigma(h, p, G, X, V, S)
        pkg.sox_check_device(h)
    check(S.cpu().numpy(), osox.sox_sigma(w.X, w.V, w.G, dtype=np.float64), prec, "after timeouts")
