"""GPU parity of single kernels at the sizes where their tiles, splits and dispatch rules
change: tile edges and remainders, the smallest sizes, both sides of every rule."""
import numpy as np
import pytest

import synth
from oracle import sox as osox
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
