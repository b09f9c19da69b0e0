"""The calls whose speed is followed, with their inputs, their work and their 64-bit results.

Every case goes through the package's public entry points, with device tensors and a handle
that the caller keeps, as a program around the library does.  The inputs are the stand-ins
that the tests and the benchmark use for molecules and solids (random Hamiltonians with a
spectrum on [-2, 2] Ha, their imaginary-time Green's functions on the Chebyshev-Lobatto grid,
normal collocation matrices, a decaying positive metric), drawn on the GPU from the seed.

``exact`` evaluates the same formulas (Sec. II B-C, III C of arXiv 2412.18829) with plain
torch / numpy in 64 bits and shares no code with the library.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2412_18829_gb300 as sox
from paper_2412_18829_gb300 import scloop

DEV = "cuda"
F64 = dict(dtype=torch.float64, device=DEV)
C128 = dict(dtype=torch.complex128, device=DEV)


def listed():
    return [
        # the small molecule: one self-energy of a few microseconds of arithmetic, where
        # launches and latency count (an inner call of a self-consistency loop)
        dict(name="sigma_small", kind="sigma", precision="f16x2", n=20, N=80, T=30, S=1, beta=100.0),
        # the mid-size unrestricted molecule: bare SOX of a whole imaginary-time grid
        dict(name="sigma_mid", kind="sigma", precision="f16x2", n=120, N=600, T=80, S=2, beta=100.0),
        # the same call on the double-precision handle (reference results, tight tolerances)
        dict(name="sigma_fp64", kind="sigma", precision="fp64", n=80, N=480, T=30, S=1, beta=100.0),
        # an uneven batch of molecules, Phi and Sigma of each (sizes of the benchmark's batch)
        dict(name="phi_batch", kind="phi_batch", precision="f16x2", sizes="57,150,79,145,75", ratio=6, T=60, beta=100.0),
        # forward and backward of Phi through autograd: a small molecule on a long grid ...
        dict(name="phi_grad_small", kind="phi_grad", precision="f16x2", n=76, N=456, T=120, S=1, beta=100.0),
        # ... and the batch's largest molecule, a few time points at a time
        dict(name="phi_grad_large", kind="phi_grad", precision="f16x2", n=298, N=1788, T=4, S=1, beta=100.0),
        # SOSEX with the static W of the same G: polarisability, W(0), self-energy
        dict(name="screened", kind="screened", precision="f16x2", n=250, N=2000, T=12, S=1, beta=100.0),
        # dynamically screened SOSEX of a molecule
        dict(name="dynamic_mid", kind="dynamic", precision="f16x2", n=120, N=600, T=80, S=1, beta=100.0),
        # dynamically screened SOSEX of a solid: a 3x3x3 mesh, some time points at a time
        dict(name="solid_333", kind="solid", precision="f16x2", mesh="3,3,3", n=26, N=300, T=8, beta=300.0),
        # a small solid mesh on a long grid
        dict(name="solid_211", kind="solid", precision="f16x2", mesh="2,1,1", n=26, N=300, T=60, beta=300.0),
        # the RPA W(i Omega) of the solid from its G, which feeds the dynamic self-energy
        dict(name="w_solid", kind="w", mesh="3,3,3", n=26, N=300, T=60, beta=300.0),
        # two iterations of the self-consistent loop around Sigma of a small molecule
        dict(name="loop_small", kind="loop", precision="fp64", n=20, N=80, T=30, S=1, beta=20.0, n_max=200),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _draw_once(rng):
    kind = rng.choice(["sigma", "sigma", "sigma_fp64", "phi_batch", "phi_grad", "phi_grad", "screened", "dynamic",
                       "solid", "w", "loop"])
    ratio = rng.uniform(4.0, 8.0)
    if kind == "sigma":
        n = _log(rng, 12, 260)
        return dict(kind="sigma", precision="f16x2", n=n, N=int(n * ratio), T=_log(rng, 8, 120), S=rng.choice([1, 2]),
                    beta=100.0)
    if kind == "sigma_fp64":
        n = _log(rng, 8, 96)
        return dict(kind="sigma", precision="fp64", n=n, N=int(n * ratio), T=_log(rng, 6, 60), S=rng.choice([1, 2]),
                    beta=100.0)
    if kind == "phi_batch":
        sizes = ",".join(str(_log(rng, 16, 180)) for _ in range(rng.randint(2, 8)))
        return dict(kind="phi_batch", precision="f16x2", sizes=sizes, ratio=rng.randint(4, 8), T=_log(rng, 8, 80),
                    beta=100.0)
    if kind == "phi_grad":
        n = _log(rng, 16, 300)
        return dict(kind="phi_grad", precision="f16x2", n=n, N=int(n * ratio), T=_log(rng, 4, 120), S=rng.choice([1, 2]),
                    beta=100.0)
    if kind == "screened":
        n = _log(rng, 24, 260)
        return dict(kind="screened", precision="f16x2", n=n, N=int(n * ratio), T=_log(rng, 8, 100), S=1, beta=100.0)
    if kind == "dynamic":
        n = _log(rng, 12, 130)
        return dict(kind="dynamic", precision="f16x2", n=n, N=int(n * ratio), T=_log(rng, 8, 80), S=rng.choice([1, 2]),
                    beta=100.0)
    mesh = rng.choice(["2,1,1", "3,1,1", "2,2,1", "2,2,2", "3,2,2", "3,3,1", "3,3,3"])
    if kind == "solid":
        n = _log(rng, 6, 30)
        return dict(kind="solid", precision="f16x2", mesh=mesh, n=n, N=int(n * rng.uniform(7.0, 12.0)), T=_log(rng, 4, 60),
                    beta=300.0)
    if kind == "w":
        n = _log(rng, 6, 30)
        return dict(kind="w", mesh=mesh, n=n, N=int(n * rng.uniform(7.0, 12.0)), T=_log(rng, 6, 60), beta=300.0)
    n = _log(rng, 4, 24)
    return dict(kind="loop", precision="fp64", n=n, N=int(n * ratio), T=_log(rng, 16, 48), S=rng.choice([1, 2]), beta=20.0,
                n_max=_log(rng, 64, 400))


def draw(rng):
    # no case dearer than the listed ones, on the GPU or in its 64-bit evaluation
    while True:
        c = _draw_once(rng)
        if _seconds(c) <= 0.25 and _exact_flops(c) <= 1.2e13:
            return c


# ----------------------------------------------------------------------------- work
def _chain_flops(n, N):
    """One (spin, tau) of the static chain: A, B and C, the Hadamard sum, projections, way back."""
    return 2.0 * N * n**3 + 4.0 * N * N * n * n + 2.0 * N * N * n + 4.0 * N * n * n + 2.0 * (N * N * n + N * n * n)


def _mesh(case):
    return tuple(int(x) for x in case["mesh"].split(","))


def work(case):
    kind, T = case["kind"], case.get("T", 0)
    if kind in ("sigma", "phi_grad", "screened", "dynamic"):
        n, N, S = case["n"], case["N"], case["S"]
        mixed = 2.0 * N * N * n * n
        flops = S * T * _chain_flops(n, N) + mixed
        io = 2.0 * S * T * n * n + N * n + N * N
        if kind == "phi_grad":     # the reverse pass: four contractions of 2 N^2 n^2 and B, C again
            flops += S * T * 12.0 * N * N * n * n + 2.0 * mixed
            io += S * T * n * n + N * n + N * N
        elif kind == "screened":   # G^PQ of every tau, Pi(0), the solve for W(0), a second mixed tensor
            flops += S * T * (2.0 * N * n * n + 2.0 * N * N * n + 2.0 * N * N) + 2.0 * N**3 + 8.0 / 3.0 * N**3 + mixed
            io += (S + 1.0) * N * N
        elif kind == "dynamic":    # transforms, the W_d product and B, C of the dynamic part
            nO = 2 * ((T - 1) // 2) + 1
            flops += S * n * (8.0 * nO * T * N * n + 4.0 * nO * N * N * n) + S * T * (4.0 * N * N * n * n + 2.0 * N * N * n)
            io += nO * N * N + 4.0 * nO * T
        return {"bytes": 8.0 * io, "flops": flops}
    if kind == "phi_batch":
        flops = io = 0.0
        for n in (int(x) for x in case["sizes"].split(",")):
            N = case["ratio"] * n
            flops += T * _chain_flops(n, N) + 2.0 * N * N * n * n
            io += 2.0 * T * n * n + N * n + N * N
        return {"bytes": 8.0 * io, "flops": flops}
    if kind == "loop":
        n, N, S, nw = case["n"], case["N"], case["S"], 2 * case["n_max"]
        # per iteration: Sigma (and once more at the end), its transform, about 50 Dyson solves on
        # every frequency, the return to tau and the Fock build
        per = S * (50 * nw * 8.0 * n**3 + 4.0 * nw * T * n * n * 2 + 4.0 * N * N * n)
        return {"bytes": 8.0 * (n * n * 3 + N * n + N * N + 2.0 * nw * T + 3.0 * S * T * n * n),
                "flops": 2 * per + 3 * (S * T * _chain_flops(n, N) + 2.0 * N * N * n * n) + S * 50 * nw * 8.0 * n**3}
    n, N, mesh = case["n"], case["N"], _mesh(case)
    k = mesh[0] * mesh[1] * mesh[2]
    nO = 2 * ((T - 1) // 2) + 1
    if kind == "solid":            # complex: 8 flops a multiply-add; B and C per pair of momenta, D by DFT over the mesh
        bc = 16.0 * k * k * N * N * n * n + 8.0 * k * k * N * N * n
        mixed = 8.0 * k * k * N * N * n * n
        stat = T * (bc + 8.0 * k * k * N * n**3 + 24.0 * k * N * n * n + 8.0 * k * N * N * n) + mixed
        dyn = T * bc + k * k * n * (16.0 * nO * T * N * n + 8.0 * nO * N * N * n)
        return {"bytes": 16.0 * (2.0 * k * T * n * n + k * N * n + k * N * N * (1 + nO)), "flops": stat + dyn}
    solve = (8.0 + 32.0 / 3.0) * N**3   # V Pi and an LU solve for N right-hand sides, half of the +-Omega pairs
    return {"bytes": 16.0 * (k * T * n * n + k * N * n + k * N * N * (1 + nO)),
            "flops": k * ((nO + 1) // 2) * solve + k * T * 8.0 * (N * n * n + N * N * n) + 8.0 * k * T * N * N * (k + nO)}


def _seconds(case):
    f = work(case)["flops"]
    rate = {"w": 6e11, "loop": 2e11, "solid": 1.2e13}.get(case["kind"], 2e14)
    return f / (7e11 if case.get("precision") == "fp64" and case["kind"] == "sigma" else rate)


def _exact_flops(case):
    return work(case)["flops"] * (1.0 if case["kind"] != "w" else 2.0)


# ----------------------------------------------------------------------------- inputs
def _tau(T, beta):
    j = np.arange(T)
    t = 0.5 * beta * (1.0 - np.cos(np.pi * j / (T - 1)))
    t[0], t[-1] = 0.0, beta
    t[T - 1 - np.arange(T // 2)] = beta - t[: T // 2]
    if T % 2:
        t[T // 2] = 0.5 * beta
    return t


def _fermi(xi, tau, beta):
    """e^{-xi tau} / (1 + e^{-beta xi}) for xi [..., n] -> [..., T, n], without overflow."""
    x, t = xi[..., None, :], tau[:, None]
    e = torch.where(x > 0, -x * t, x * (beta - t))
    return torch.exp(e) / (1.0 + torch.exp(-beta * x.abs()))


def _spectrum(h):
    """Eigenpairs of h with the spectrum mapped to [-2, 2] Ha."""
    e, u = torch.linalg.eigh(h)
    return -2.0 + (e - e[0]) * 4.0 / (e[-1] - e[0]), u


def _metric(N, gen, kw):
    z = torch.randn(N, N, generator=gen, **kw)
    z = z / torch.linalg.vector_norm(z, dim=0) / (1.0 + torch.arange(N, **F64))
    return z @ z.mH


def _molecule(n, N, T, S, beta, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    a = torch.randn(n, n, generator=gen, **F64)
    e, u = _spectrum(0.5 * (a + a.T))
    mu = float(0.5 * (e[n // 2 - 1] + e[n // 2]))
    h = (u * e) @ u.T
    tau = torch.from_numpy(_tau(T, beta)).to(DEV)
    G = torch.empty(S, 1, T, n, n, **F64)
    for s in range(S):
        if S == 2:               # unrestricted: the first orbitals shifted up or down
            m = min(10, n)
            d = torch.zeros(n, **F64)
            d[:m] = -0.05 if s == 0 else 0.05
            e, u = torch.linalg.eigh(h + torch.diag(d))
        f = _fermi(e - mu, tau, beta)
        G[s, 0] = -(u * f[:, None, :]) @ u.T
    X = torch.randn(1, N, n, generator=gen, **F64) / math.sqrt(n)
    return dict(h0=h, G=G, X=X, V=_metric(N, gen, F64)[None].contiguous())


def _solid(n, N, T, mesh, beta, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    ks = np.stack(np.meshgrid(*[np.arange(d) for d in mesh], indexing="ij"), axis=-1).reshape(-1, 3)
    kv = torch.from_numpy(2.0 * np.pi * ks / np.asarray(mesh)).to(DEV)
    nk = len(ks)
    a = torch.randn(n, n, generator=gen, **F64)
    e, u = _spectrum(0.5 * (a + a.T))
    H = ((u * e) @ u.T).to(torch.complex128).repeat(nk, 1, 1)
    for d in range(3):
        t = torch.randn(n, n, generator=gen, **F64) * (0.1 / math.sqrt(n))
        ph = torch.exp(1j * kv[:, d])[:, None, None]
        H = H + t * ph + t.T * ph.conj()
    e, u = torch.linalg.eigh(0.5 * (H + H.mH))
    lv = torch.sort(e.reshape(-1)).values
    mu = float(0.5 * (lv[n * nk // 2 - 1] + lv[n * nk // 2]))
    f = _fermi(e - mu, torch.from_numpy(_tau(T, beta)).to(DEV), beta)
    G = (-(u[:, None] * f[:, :, None, :]) @ u.mH[:, None])[None].contiguous()
    x0 = torch.randn(N, n, generator=gen, **C128) / math.sqrt(n)
    r = torch.rand(N, 3, generator=gen, **F64)
    X = (x0 * torch.exp(1j * (kv @ r.T))[:, :, None]).contiguous()
    V = torch.empty(nk, N, N, **C128)
    done = set()
    for q in range(nk):
        m = np.mod(-ks[q], mesh)
        p = int((m[0] * mesh[1] + m[1]) * mesh[2] + m[2])
        if q in done:
            continue
        V[q] = _metric(N, gen, C128 if p != q else F64)
        V[p] = V[q].conj()
        done |= {q, p}
    return dict(G=G, X=X, V=V)


def _bosonic(T, beta):
    """tau -> i Omega and back on the grid's interpolant, Omega_m = 2 pi m / beta."""
    tau, M = _tau(T, beta), (T - 1) // 2
    om = 2.0 * np.pi * np.arange(-M, M + 1) / beta
    x, wg = np.polynomial.legendre.leggauss(512)
    s, wg = 0.5 * beta * (x + 1.0), 0.5 * beta * wg
    bw = (-1.0) ** np.arange(T)
    bw[[0, -1]] *= 0.5
    r = bw / (s[:, None] - tau)
    Tf = (np.exp(1j * om[:, None] * s) * wg) @ (r / r.sum(axis=1, keepdims=True))
    Ti = np.exp(-1j * tau[:, None] * om) / beta
    return om, torch.from_numpy(Tf).to(DEV), torch.from_numpy(Ti).to(DEV)


def _fermionic(T, beta, n_max):
    """tau -> i w on the grid's interpolant, w_m = (2m + 1) pi / beta."""
    tau, om = _tau(T, beta), (2 * np.arange(-n_max, n_max) + 1) * np.pi / beta
    x, wg = np.polynomial.legendre.leggauss(16)
    edges = np.linspace(0.0, beta, 2 * n_max + 2)
    half = 0.5 * np.diff(edges)
    s = (edges[:-1, None] + half[:, None] * (x + 1.0)).ravel()
    ws = (half[:, None] * wg).ravel()
    bw = (-1.0) ** np.arange(T)
    bw[[0, -1]] *= 0.5
    r = bw / (s[:, None] - tau)
    return om, (np.exp(1j * om[:, None] * s) * ws) @ (r / r.sum(axis=1, keepdims=True))


def _pole_screening(V, om, seed):
    """W - v of a single plasmon pole: -1/2 w_p^2 / (Omega^2 + w_p^2) V D V / |V|, [q][Omega][N][N]."""
    gen = torch.Generator(device=DEV).manual_seed(seed + 1)
    d = 0.5 + torch.rand(V.shape[-1], generator=gen, **F64)
    vdv = (V * d) @ V
    f = torch.from_numpy(-0.125 / (om**2 + 0.25)).to(DEV) / torch.linalg.matrix_norm(V[0], 2)
    return (f[None, :, None, None] * vdv[:, None]).contiguous()


def _weights(T, beta):
    return sox.sox_tau_grid(T, beta)[1]


def _inputs(case, seed):
    """The tensors of a case (no library call but the grid's weights)."""
    kind, T, beta = case["kind"], case["T"], case["beta"]
    if kind == "phi_batch":
        sizes = [int(x) for x in case["sizes"].split(",")]
        return dict(mol=[_molecule(n, case["ratio"] * n, T, 1, beta, seed * 64 + i) for i, n in enumerate(sizes)])
    if kind in ("solid", "w"):
        d = _solid(case["n"], case["N"], T, _mesh(case), beta, seed)
        om, d["Tf"], d["Ti"] = _bosonic(T, beta)
        if kind == "solid":
            d["Wd"] = _pole_screening(d["V"], om, seed)
        return d
    d = _molecule(case["n"], case["N"], T, case["S"], beta, seed)
    if kind == "dynamic":
        om, d["Tf"], d["Ti"] = _bosonic(T, beta)
        d["Wd"] = _pole_screening(d["V"], om, seed)[0]
    return d


def prepare(case, seed):
    kind, T, beta = case["kind"], case["T"], case["beta"]
    d = _inputs(case, seed)
    s = dict(kind=kind, handle=sox.Handle(case.get("precision", "fp64")))
    if kind == "phi_batch":
        m = d["mol"]
        s.update(p=[sox.problem(x["G"].shape[-1], x["V"].shape[-1], T, 1, beta) for x in m], G=[x["G"] for x in m],
                 X=[x["X"] for x in m], V=[x["V"] for x in m], w=[torch.from_numpy(_weights(T, beta)).to(DEV) for _ in m],
                 phi=[torch.empty(1, **F64) for _ in m], Sigma=[torch.empty_like(x["G"]) for x in m])
        return s
    if kind in ("solid", "w"):
        s.update(d, p=sox.problem(case["n"], case["N"], T, 1, beta, nk=_mesh(case), dtype=1), nO=d["Tf"].shape[0])
        if kind == "solid":
            s["Sigma"] = torch.empty_like(d["G"])
        else:
            s["Wd"] = torch.empty(d["V"].shape[0], s["nO"], case["N"], case["N"], **C128)
        return s
    s.update(d, p=sox.problem(case["n"], case["N"], T, case["S"], beta))
    if kind in ("sigma", "dynamic", "screened"):
        s["Sigma"] = torch.empty_like(d["G"])
    if kind == "dynamic":
        s["nO"] = d["Tf"].shape[0]
    if kind in ("phi_grad", "screened", "loop"):
        s["w"] = torch.from_numpy(_weights(T, beta)).to(DEV)
    if kind == "phi_grad":
        for k in ("G", "X", "V"):
            s[k].requires_grad_(True)
    if kind == "screened":
        s["Pi"], s["W0"] = torch.empty(1, case["N"], case["N"], **F64), torch.empty(1, case["N"], case["N"], **F64)
    if kind == "loop":
        om, Tw = _fermionic(T, beta, case["n_max"])
        s.update(V=0.3 * s["V"].contiguous(), om=torch.from_numpy(om).to(DEV), Tw=torch.from_numpy(Tw).to(DEV),
                 tau=torch.from_numpy(_tau(T, beta)).to(DEV), n_elec=float(case["n"] // 2) * case["S"])
    return s


def run(s):
    kind, h, p = s["kind"], s["handle"], s["p"]
    if kind == "sigma":
        sox.sox_sigma(h, p, s["G"], s["X"], s["V"], s["Sigma"])
        return s["Sigma"]
    if kind == "phi_batch":
        sox.phi_sox_batch(h, p, s["G"], s["X"], s["V"], s["w"], s["phi"], s["Sigma"])
        return {"phi": s["phi"], "Sigma": s["Sigma"]}
    if kind == "phi_grad":
        phi = sox.PhiSOX.apply(s["G"], s["X"], s["V"], s["w"], h, p)
        dG, dX, dV = torch.autograd.grad(phi.sum(), (s["G"], s["X"], s["V"]))
        return {"phi": phi.detach(), "dG": dG, "dX": dX, "dV": dV}
    if kind == "screened":
        sox.sox_pi0(h, p, s["G"], s["X"], s["w"], s["Pi"])
        sox.sox_w_static(h, p, s["V"], s["Pi"], s["W0"])
        sox.sosex_static_sigma(h, p, s["G"], s["X"], s["V"], s["W0"], s["Sigma"])
        return {"Pi": s["Pi"], "W0": s["W0"], "Sigma": s["Sigma"]}
    if kind in ("dynamic", "solid"):
        sox.sosex_dynamic_sigma(h, p, s["G"], s["X"], s["V"], s["Wd"], s["Tf"], s["Ti"], s["nO"], s["Sigma"])
        return s["Sigma"]
    if kind == "w":
        sox.sox_w_dynamic(h, p, s["G"], s["X"], s["V"], s["Tf"], s["nO"], s["Wd"])
        return s["Wd"]
    r = scloop.run(h, p, s["h0"], s["X"], s["V"], s["n_elec"], s["om"], s["Tw"], s["tau"], s["w"], max_iter=2)
    return {"G": r.G_tau, "mu": r.mu, "gamma": r.gamma, "Sigma_hf": r.sigma_hf, "Sigma": r.sigma_tau, "E": r.energies,
            "change": r.change}


# ----------------------------------------------------------------------------- 64-bit results
def _pairs(X):
    """X_Qq X_Qs, [N][n n]."""
    N, n = X.shape
    return (X[:, :, None] * X[:, None, :]).reshape(N, n * n)


def _d_step(Gj, Gm, X, U1, U2):
    """D_PR of one time from the mixed tensors U1, U2 [N][n][n] (Sec. II C)."""
    N, n = X.shape
    GR, GW = X @ Gj, X @ Gj.T
    A = (U1.reshape(N * n, n) @ Gm).reshape(N, n, n).permute(2, 0, 1)     # [v][P][q]
    D = torch.zeros(N, N, **F64)
    step = max(1, int(2e9 // (8 * N * N)))
    for v in range(0, n, step):
        B = A[v:v + step] @ GR.T                                           # [v][P][R]
        C = GW @ U2[:, v:v + step].permute(1, 2, 0)
        D = D + (B * C).sum(0)
    return D


def _sigma(G, X, V1, V2):
    S, _, T, n, _ = G.shape
    N = X.shape[0]
    U1 = (V1 @ _pairs(X)).reshape(N, n, n)
    U2 = U1 if V2 is V1 else (V2 @ _pairs(X)).reshape(N, n, n)
    out = torch.empty_like(G)
    for s in range(S):
        for j in range(T):
            out[s, 0, j] = -(X.T @ _d_step(G[s, 0, j], -G[s, 0, T - 1 - j], X, U1, U2).T @ X)
    return out


def _phi(Sigma, G, w):
    return 0.25 * torch.einsum("j,sjtr,sjrt->s", w, Sigma[:, 0], -G[:, 0].flip(1))


def _phi_grads(d, w):
    G, X, V = (d[k].clone().requires_grad_(True) for k in ("G", "X", "V"))
    S, _, T, n, _ = G.shape
    N = X.shape[1]
    U = V[0] @ _pairs(X[0])
    Ud = U.detach().reshape(N, n, n).requires_grad_(True)
    phi = torch.zeros(S, **F64)
    for s in range(S):
        for j in range(T):
            Gm = -G[s, 0, T - 1 - j]
            Sg = -(X[0].T @ _d_step(G[s, 0, j], Gm, X[0], Ud, Ud).T @ X[0])
            f = 0.25 * w[j] * (Sg * Gm.T).sum()
            f.backward()
            phi[s] += f.detach()
    U.backward(Ud.grad.reshape(N, n * n))
    return {"phi": phi, "dG": G.grad, "dX": X.grad, "dV": V.grad}


def _dynamic(d, nO):
    G, X, V = d["G"], d["X"][0], d["V"][0]
    S, _, T, n, _ = G.shape
    N = X.shape[0]
    out = _sigma(G, X, V, V)
    U2 = (V @ _pairs(X)).reshape(N, n, n)
    Fr, Fi, Ir, Ii = d["Tf"].real, d["Tf"].imag, d["Ti"].real, d["Ti"].imag
    for s in range(S):
        g, gm = G[s, 0], -G[s, 0].flip(0)
        GQu = X @ g.transpose(1, 2)            # G_uQ(tau_j) as [j][Q][u]
        GQv = X @ gm                           # [j][Q][v]
        GW = X @ g.transpose(1, 2)             # G_wP as [j][P][w]
        D = torch.zeros(T, N, N, **F64)
        for v in range(n):
            GG = (GQu * GQv[:, :, v, None]).reshape(T, N * n)
            Ar = d["Wd"] @ (Fr @ GG).reshape(nO, N, n)
            Ai = d["Wd"] @ (Fi @ GG).reshape(nO, N, n)
            At = (Ir @ Ar.reshape(nO, N * n) - Ii @ Ai.reshape(nO, N * n)).reshape(T, N, n)
            D += (At @ X.T) * (GW @ U2[:, v].T)
        out[s, 0] -= X.T @ D.transpose(1, 2) @ X
    return out


def _tables(mesh):
    g = np.stack(np.meshgrid(*[np.arange(x) for x in mesh], indexing="ij"), axis=-1).reshape(-1, 3)

    def at(m):
        m = np.mod(m, mesh)
        return int((m[0] * mesh[1] + m[1]) * mesh[2] + m[2])

    return ([[at(a + b) for b in g] for a in g], [[at(a - b) for b in g] for a in g])


def _solid_sigma(d, mesh, nO):
    G, X, V, Wd, Tf, Ti = d["G"][0], d["X"], d["V"], d["Wd"], d["Tf"], d["Ti"]
    nk, T, n, _ = G.shape
    N = X.shape[1]
    _, sub = _tables(mesh)
    g, gm = G, -G.flip(1)
    GR = X[:, None] @ g                                    # [k][j][R][q]
    GQu = X.conj()[:, None] @ g.transpose(2, 3)            # G_uQ as [k][j][Q][u]
    GW = GQu                                               # G_wP as [k][j][P][w]
    GQv = X[:, None] @ gm                                  # [k][j][Q][v]
    M = torch.empty(nk, nk, N, n, n, **C128)               # U^{q,k}[P][a][b]
    for q in range(nk):
        for k in range(nk):
            M[q, k] = (V[q] @ (X[sub[k][q]].conj()[:, :, None] * X[k][:, None, :]).reshape(N, n * n)).reshape(N, n, n)
    D = torch.zeros(T, nk, N, N, **C128)
    for v in range(n):
        for j0 in range(0, T, 4):
            js = slice(j0, min(T, j0 + 4))
            nj = js.stop - js.start
            c = torch.empty(nk, nk, nj, N, N, **C128)      # [k_s][k_w]: C of transfer k_w - k_s
            for kw in range(nk):
                for ks in range(nk):
                    c[ks, kw] = GW[kw, js] @ M[sub[kw][ks], kw][:, v].T
            ch = torch.fft.fftn(c.reshape((nk,) + mesh + (nj, N, N)), dim=(1, 2, 3))
            del c
            b = torch.empty(nk, nk, nj, N, N, **C128)      # [k_s][j = k_s - q1]: B of transfer q1
            for ks in range(nk):
                for j in range(nk):
                    q1 = sub[ks][j]
                    A = torch.einsum("Pqs,tsx->tPqx", M[q1, ks], gm[ks, js][:, :, v:v + 1])[..., 0]
                    GG = (GQu[j] * GQv[ks][:, :, v, None]).reshape(T, N * n)
                    Aw = Wd[q1] @ (Tf @ GG).reshape(nO, N, n)
                    At = (Ti[js] @ Aw.reshape(nO, N * n)).reshape(nj, N, n)
                    # slot j holds k_q = k_s - q1; the sum over q1 at fixed k_w - k and k_s
                    b[ks, q1] = A @ GR[j, js].transpose(1, 2) + At @ X[j].T
            # D[k] = sum_{ks} sum_{q1} c[ks][k + q1] b[ks][q1]
            bh = torch.fft.ifftn(b.reshape((nk,) + mesh + (nj, N, N)), dim=(1, 2, 3))
            del b
            D[js] += (torch.fft.ifftn((ch * bh).sum(0), dim=(0, 1, 2)).reshape(nk, nj, N, N) * nk).transpose(0, 1)
            del ch, bh
    D = D / nk**2
    out = torch.empty_like(G)
    for k in range(nk):
        out[k] = -(X[k].mH @ D[:, k].transpose(1, 2) @ X[k])
    return out[None]


def _w_solid(d, mesh, nO):
    G, X, V, Tf = d["G"][0], d["X"], d["V"], d["Tf"]
    nk, T, n, _ = G.shape
    N = X.shape[1]
    add, _ = _tables(mesh)
    gp = X[:, None] @ G @ X.mH[:, None]                    # [k][j][P][Q]
    gm = -gp.flip(1)
    W = torch.empty(nk, nO, N, N, **C128)
    one = torch.eye(N, **C128)
    for q in range(nk):
        pi = torch.zeros(T, N, N, **C128)
        for k in range(nk):
            pi += gp[add[k][q]] * gm[k].transpose(1, 2)
        pi = (Tf @ pi.reshape(T, N * N)).reshape(nO, N, N) / nk
        W[q] = torch.linalg.solve(one - V[q] @ pi, V[q].expand(nO, N, N)) - V[q]
    return W


def _loop(case, d):
    h0, X, V = (d[k].cpu().numpy() for k in ("h0", "X", "V"))
    X, V = X[0], 0.3 * V[0]
    n, T, S, beta = case["n"], case["T"], case["S"], case["beta"]
    tau, w = _tau(T, beta), _weights(T, beta)
    om, Tw = _fermionic(T, beta, case["n_max"])
    iw, one = 1j * om[:, None, None], np.eye(n)
    n_elec = float(n // 2) * S
    img = (-0.5 * np.ones(T), (2 * tau - beta) / 4, tau * (beta - tau) / 4)

    def green(mu, F, Siw, Stau, at):
        R = np.linalg.inv((iw + mu) * one - F - Siw)
        a = F - mu * one
        c = (one, a, a @ a - (Stau[-1] + Stau[0]))
        for k in range(3):
            R = R - c[k] / iw ** (k + 1)
        ph = np.exp(-1j * tau[at, None] * om) / beta
        return np.einsum("tw,wpq->tpq", ph, R).real + sum(img[k][at][:, None, None] * c[k] for k in range(3))

    def find(Fs, Siws, Staus):
        lo, hi = -50.0, 50.0
        for _ in range(200):
            if hi - lo < 1e-13:
                break
            mid = 0.5 * (lo + hi)
            cnt = sum(-np.trace(green(mid, F, a, b, np.array([T - 1]))[0]) for F, a, b in zip(Fs, Siws, Staus))
            lo, hi = (mid, hi) if cnt < n_elec else (lo, mid)
        return 0.5 * (lo + hi)

    def fock(gam):
        dQ = np.einsum("Qr,Qs,rs->Q", X, X, gam.sum(0), optimize=True)
        J = np.einsum("Pp,Pq,P->pq", X, X, V @ dQ, optimize=True)
        return np.stack([J - X.T @ (V * (X @ g @ X.T)) @ X for g in gam])

    def sigma(G):
        Gd = torch.from_numpy(np.ascontiguousarray(G[:, None])).to(DEV)
        Xd, Vd = torch.from_numpy(X).to(DEV), torch.from_numpy(V).to(DEV)
        return _sigma(Gd, Xd, Vd, Vd)[:, 0].cpu().numpy()

    z, zw, every = np.zeros((T, n, n)), np.zeros((len(om), n, n), complex), np.arange(T)
    mu = find([h0] * S, [zw] * S, [z] * S)
    G = np.stack([green(mu, h0, zw, z, every) for _ in range(S)])
    for _ in range(2):
        gam = np.stack([-g[-1].T for g in G])
        F = h0 + fock(gam)
        St = sigma(G)
        Sw = [(Tw @ St[s].reshape(T, n * n)).reshape(-1, n, n) for s in range(S)]
        mu = find(F, Sw, St)
        new = np.stack([green(mu, F[s], Sw[s], St[s], every) for s in range(S)])
        change = float(np.abs(new - G).max())
        G = 0.5 * G + 0.5 * new
    gam = np.stack([-g[-1].T for g in G])
    hf, St = fock(gam), sigma(G)
    E = np.array([np.sum((h0 + 0.5 * hf) * gam),
                  -sum(np.einsum("j,jpq,jqp->", w, St[s][::-1], G[s]) for s in range(S))])
    return {"G": G, "mu": mu, "gamma": gam, "Sigma_hf": hf, "Sigma": St, "E": E, "change": change}


def exact(case, seed):
    kind = case["kind"]
    if _exact_flops(case) > 2.2e13:
        return None
    d = _inputs(case, seed)
    if kind == "sigma":
        return _sigma(d["G"], d["X"][0], d["V"][0], d["V"][0])
    w = torch.from_numpy(_weights(case["T"], case["beta"])).to(DEV)
    if kind == "phi_batch":
        S = [_sigma(m["G"], m["X"][0], m["V"][0], m["V"][0]) for m in d["mol"]]
        return {"phi": [_phi(x, m["G"], w) for x, m in zip(S, d["mol"])], "Sigma": S}
    if kind == "phi_grad":
        return _phi_grads(d, w)
    if kind == "screened":
        G, X, V = d["G"], d["X"][0], d["V"][0]
        gp = X @ G[0, 0] @ X.T
        Pi = -(w[:, None, None] * gp * gp.flip(0).transpose(1, 2)).sum(0)
        W0 = torch.linalg.solve(torch.eye(len(V), **F64) - V @ Pi, V)
        return {"Pi": Pi[None], "W0": W0[None], "Sigma": _sigma(G, X, W0, V)}
    if kind == "dynamic":
        return _dynamic(d, d["Tf"].shape[0])
    if kind == "solid":
        return _solid_sigma(d, _mesh(case), d["Tf"].shape[0])
    if kind == "w":
        return _w_solid(d, _mesh(case), d["Tf"].shape[0])
    return _loop(case, d)
