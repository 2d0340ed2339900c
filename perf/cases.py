"""Performance cases: calls of the public solver API at the sizes, precisions and options it is used
with, from a 64-site chain to N = 8192.

One pass is what a program repeats per Hamiltonian: it loads H0 (and the perturbations H1) and
asks for the density matrix with a response, a gradient or a free energy. Inputs are made on the
GPU from the seed: the open chain, disordered cubic lattices (orders of the sites follow the
lattice), banded random matrices and disordered clusters that the tests and bench.py use.

FP64 solves hand on FP64 results. FP32 and mixed solves compute FP32-accurate numbers (bars 1e-5
and 1e-6), which the programs here keep as FP32 matrices.
"""
import math

import numpy as np
import torch

import paper_1503_07037_gb300 as cdmpt

# ------------------------------------------------------------------------------- the cases


def listed():
    return [
        # first contact and unit tests of a user's model: the 64-site chain in FP64; all latency
        dict(name="chain64-fp64", kind="solve", model="chain", precision="fp64", N=64, beta=10.0,
             n=12, D=1),
        # a small periodic cell with its full dipole response (three directions), mixed precision
        dict(name="lattice512-mixed-xyz", kind="solve", model="lattice", precision="mixed",
             Lx=8, Ly=8, Lz=8, beta=20.0, n=14, D=3),
        # FP32 at an odd size: rows that are no multiple of any tile, a ragged last tile
        dict(name="lattice1001-fp32", kind="solve", model="lattice", precision="fp32",
             Lx=13, Ly=11, Lz=7, beta=20.0, n=14, D=1),
        # the reference-accuracy path at an ordinary size (FP64 products on the tensor cores)
        dict(name="lattice2048-fp64", kind="solve", model="lattice", precision="fp64",
             Lx=16, Ly=16, Lz=8, beta=20.0, n=14, D=1),
        # the 16^3 lattice: the mixed default, and FP32 at a low temperature
        dict(name="lattice4096-mixed", kind="solve", model="lattice", precision="mixed",
             Lx=16, Ly=16, Lz=16, beta=20.0, n=14, D=1),
        dict(name="lattice4096-fp32-cold", kind="solve", model="lattice", precision="fp32",
             Lx=16, Ly=16, Lz=16, beta=80.0, n=14, D=1),
        # the largest: the N = 8192 banded system of the headline benchmark
        dict(name="banded8192-mixed", kind="solve", model="banded", precision="mixed", N=8192,
             beta=20.0, n=14, D=1),
        # fitting a Hamiltonian: loss of P0 back to H0 through the adjoint, sqrt(n) checkpoints
        dict(name="adjoint2048-fp32", kind="adjoint", model="lattice", precision="fp32",
             Lx=16, Ly=16, Lz=8, beta=20.0, n=16, ckpt=True),
        # gradient of the polarizability (second-order response), FP32
        dict(name="alpha-grad1000-fp32", kind="alpha_grad", model="lattice", precision="fp32",
             Lx=10, Ly=10, Lz=10, beta=20.0, n=14, D=1),
        # Mermin free energy as a loss with its gradient, FP64, ragged N = 343
        dict(name="free-energy343-fp64", kind="free_energy", model="lattice", precision="fp64",
             Lx=7, Ly=7, Lz=7, beta=20.0, n=14),
        # a batch of uneven clusters, three dipole directions each, at one temperature
        dict(name="batch24-mixed", kind="batch", precision="mixed", B=24, nmin=128, nmax=1536,
             pick=1, beta=20.0, n=12, D=3),
        # self-consistent charges and their linear response in a non-orthogonal basis (host arrays)
        dict(name="scc120-fp64", kind="scc", precision="fp64", N=120, beta=20.0, n=14),
    ]


def _loguniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _lattice_dims(rng, lo, hi):
    """Three edges of about equal length with a product of about a log-uniform N in lo..hi."""
    edge = _loguniform(rng, lo, hi) ** (1.0 / 3.0)
    d = [max(3, int(round(edge * rng.uniform(0.8, 1.25)))) for _ in range(2)]
    N = max(lo, min(hi, edge ** 3))
    d.append(max(3, min(int(round(N / (d[0] * d[1]))), hi // (d[0] * d[1]))))
    return dict(model="lattice", Lx=d[0], Ly=d[1], Lz=d[2])


def draw(rng):
    """One more case: solves twice as often as the derivatives, batches and charge loops."""
    kind = rng.choice(["solve"] * 5 + ["adjoint", "alpha_grad", "free_energy", "batch", "scc"])
    beta = round(math.exp(rng.uniform(math.log(5.0), math.log(80.0))), 3)
    if kind == "solve":
        precision = rng.choice(["fp64", "fp32", "mixed"])
        top = {"fp64": 2048, "fp32": 4096, "mixed": 6000}[precision]
        model = rng.choice(["chain", "lattice", "lattice", "banded"])
        c = dict(kind=kind, precision=precision, beta=beta, n=14)
        if model == "lattice":
            c.update(_lattice_dims(rng, 64, top), D=rng.choice([1, 1, 3]))
        else:
            lo = 64 if model == "chain" else 300
            c.update(model=model, N=_loguniform(rng, lo, top), D=1)
        return c
    if kind == "adjoint":
        return dict(kind=kind, precision=rng.choice(["fp32", "fp64"]), beta=beta, n=16,
                    ckpt=rng.random() < 0.5, **_lattice_dims(rng, 64, 2048))
    if kind == "alpha_grad":
        return dict(kind=kind, precision=rng.choice(["fp32", "fp64", "mixed"]), beta=beta, n=14,
                    D=rng.choice([1, 2]), **_lattice_dims(rng, 64, 1100))
    if kind == "free_energy":
        return dict(kind=kind, precision=rng.choice(["fp32", "fp64"]), beta=beta, n=14,
                    **_lattice_dims(rng, 64, 1500))
    if kind == "batch":
        return dict(kind=kind, precision=rng.choice(["fp32", "mixed"]), B=rng.randint(4, 24),
                    nmin=128, nmax=_loguniform(rng, 300, 1536), pick=rng.randint(2, 1 << 20),
                    beta=20.0, n=12, D=3)
    return dict(kind=kind, precision="fp64", N=_loguniform(rng, 48, 180), beta=20.0, n=14)


# ------------------------------------------------------------------------------- inputs


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _f64(shape, g, normal=False):
    f = torch.randn if normal else torch.rand
    return f(shape, generator=g, dtype=torch.float64, device="cuda")


def _dipoles(coords):
    return torch.stack([torch.diag(x - x.mean()) for x in coords])


#: On-site level: energies are counted from the vacuum, a few hoppings above the band's centre.
LEVEL = -2.0


def _hamiltonian(case, seed):
    """(H0, H1): N x N and D x N x N float64 CUDA tensors."""
    H0, H1 = _centred(case, seed)
    H0.diagonal().add_(LEVEL)
    return H0, H1


def _centred(case, seed):
    g = _gen(seed)
    if case["model"] == "lattice":
        L = (case["Lx"], case["Ly"], case["Lz"])
        N = L[0] * L[1] * L[2]
        i = torch.arange(N, device="cuda")
        c = [i // (L[1] * L[2]), i // L[2] % L[1], i % L[2]]
        H0 = torch.diag(0.3 * _f64((N,), g, normal=True))
        for a in range(3):   # one bond to the next site along each axis, periodic
            nb = list(c)
            nb[a] = (c[a] + 1) % L[a]
            j = (nb[0] * L[1] + nb[1]) * L[2] + nb[2]
            hop = -(1.0 + 0.1 * (2.0 * _f64((N,), g) - 1.0))
            H0.index_put_((i, j), hop, accumulate=True)
            H0.index_put_((j, i), hop, accumulate=True)
        return H0, _dipoles([x.double() for x in c][:case.get("D", 1)])
    N = case["N"]
    x = torch.arange(N, dtype=torch.float64, device="cuda")
    if case["model"] == "chain":
        off = torch.full((N - 1,), -1.0, dtype=torch.float64, device="cuda")
        H0 = torch.diag(2.0 * _f64((N,), g) - 1.0) + torch.diag(off, 1) + torch.diag(off, -1)
    else:   # banded: |i - j| <= 64, entries N(0, 1) / 8
        H0 = torch.triu(_f64((N, N), g, normal=True).mul_(0.125))
        H0 = torch.tril(H0, 64)
        H0 = H0 + torch.triu(H0, 1).T
    return H0, _dipoles([x])


def _cluster_sizes(case):
    """The sizes are part of the workload and do not change with the seed."""
    r = np.random.default_rng(case["pick"])
    return [int(v) for v in r.integers(case["nmin"], case["nmax"] + 1, size=case["B"])]


def _cluster(N, g):
    pos = N ** (1.0 / 3.0) * _f64((N, 3), g)
    eps = 0.3 * _f64((N,), g, normal=True)
    r = (pos[:, None, :] - pos[None, :, :]).square().sum(-1).sqrt()
    H0 = torch.where((r < 2.5) & (r > 0.0), -torch.exp(-2.0 * (r - 1.0)), 0.0)
    H0 = 0.5 * (H0 + H0.T)
    H0.diagonal().copy_(eps + LEVEL)
    return H0, _dipoles([pos[:, a] for a in range(3)])


def _scc_model(N, seed):
    """Non-orthogonal cluster: S, F, one Mulliken dipole, the charge kernel and reference charges."""
    g = _gen(seed)
    pos = N ** (1.0 / 3.0) * _f64((N, 3), g)
    eps = 0.3 * _f64((N,), g, normal=True)
    r2 = (pos[:, None, :] - pos[None, :, :]).square().sum(-1)
    r2 = 0.5 * (r2 + r2.T)
    S = 0.3 * torch.exp(-r2 / 1.28)
    S.diagonal().add_(0.7)
    F = -4.0 * S
    F.diagonal().copy_(eps)
    x = pos[:, 0] - pos[:, 0].mean()
    h1 = (0.5 * S * (x[:, None] + x[None, :]))[None]
    gamma = 0.5 * torch.exp(-r2 / 2.0)
    return [t.cpu().numpy() for t in (S, F, h1, gamma)] + [np.ones(N)]


def _sym_normal(N, g):
    G = _f64((N, N), g, normal=True)
    return 0.5 * (G + G.T)


def prepare(case, seed):
    """The inputs on the GPU and the handle (or batch) that a program keeps for this size."""
    kind = case["kind"]
    s = {"case": dict(case)}
    if kind == "batch":
        # one set of systems, solved for its temperature: the batch holds the Hamiltonians
        g = _gen(seed)
        s["sizes"] = _cluster_sizes(case)
        sys_ = [_cluster(N, g) for N in s["sizes"]]
        s["batch"] = cdmpt.Batch(s["sizes"], case["D"], precision=case["precision"])
        s["batch"].set_H([h0.cpu().numpy() for h0, _ in sys_], [h1.cpu().numpy() for _, h1 in sys_],
                         case["n"])
        return s
    if kind == "scc":
        S, s["F"], s["h1"], s["gamma"], s["q0"] = _scc_model(case["N"], seed)
        s["handle"] = cdmpt.Handle(precision=case["precision"])
        s["handle"].set_overlap(S)
        return s
    s["H0"], s["H1"] = _hamiltonian(case, seed)
    s["handle"] = cdmpt.Handle(precision=case["precision"],
                               ckpt_stride="sqrt" if case.get("ckpt") else 0)
    if kind == "adjoint":
        s["G"] = _sym_normal(s["H0"].shape[0], _gen(seed + 1))
    if kind != "solve":
        s["H0"].requires_grad_(True)
    return s


# ------------------------------------------------------------------------------- the pass


def _keep(case, *tensors):
    """Results as the program keeps them: FP64 from FP64 solves, FP32 from the others."""
    if case["precision"] == "fp64":
        return tensors
    return tuple(t.float() if isinstance(t, torch.Tensor) else np.asarray(t, dtype=np.float32)
                 for t in tensors)


def run(state):
    case = state["case"]
    kind, n, beta = case["kind"], case["n"], case["beta"]
    if kind == "batch":
        sizes = state["sizes"]
        r = state["batch"].solve([beta] * len(sizes), [float(N // 2) for N in sizes], n)
        pot = np.concatenate([r["mu"][:, None], r["mu1"]], axis=1)
        return _keep(case, *r["P0"], *r["P1"], pot, r["alpha"])
    if kind == "scc":
        r = state["handle"].scc_solve(state["F"], state["h1"], state["gamma"], beta,
                                      float(case["N"] // 2), n, q0=state["q0"])
        pot = np.concatenate([[r["mu"]], r["mu1"]])
        return r["D0"], r["D1"], pot, r["omega1"], r["omega2"]
    h, H0 = state["handle"], state["H0"]
    nocc = H0.shape[0] / 2.0
    if kind == "solve":
        h.set_H(H0, state["H1"])
        r = h.solve(beta, nocc, n)
        pot = np.concatenate([[r["mu"]], r["mu1"]])
        return _keep(case, r["P0"], r["P1"], pot, h.polarizability())
    if kind == "adjoint":
        P0 = cdmpt.DensityMatrix.apply(H0, beta, nocc, n, h)
        (grad,) = torch.autograd.grad(P0, H0, state["G"])
        return _keep(case, P0.detach(), grad)
    if kind == "alpha_grad":
        alpha = cdmpt.Polarizability.apply(H0, state["H1"], beta, nocc, n, h)
        (grad,) = torch.autograd.grad(alpha.sum(), H0)
        return _keep(case, alpha.detach(), grad)
    omega = cdmpt.FreeEnergy.apply(H0, beta, nocc, n, h)
    (grad,) = torch.autograd.grad(omega, H0)
    return _keep(case, omega.detach(), grad)


def _size(case):
    return case["Lx"] * case["Ly"] * case["Lz"] if case.get("model") == "lattice" else case["N"]


def work(case):
    """Inputs read once and outputs written once; the products that no form of the recursion does
    without: per step the square of the iterate and the new iterate (symmetric results, N^3 each)
    and two products per direction of the response or of the gradient (2 N^3 each)."""
    kind, n = case["kind"], case["n"]
    out = 8 if case["precision"] == "fp64" else 4

    def one(N, D):
        return N * N * (1 + D) * (8.0 + out), n * (2.0 + 4.0 * D) * float(N) ** 3

    if kind == "batch":
        pairs = [one(N, case["D"]) for N in _cluster_sizes(case)]
        return {"bytes": sum(p[0] for p in pairs), "flops": sum(p[1] for p in pairs)}
    N = _size(case)
    if kind == "solve":
        b, f = one(N, case["D"])
    elif kind == "adjoint":
        b, f = one(N, 1)
    elif kind == "alpha_grad":   # orders 1 and 2 per direction, order 1 once for alpha
        b, f = one(N, case["D"])
        f += n * 8.0 * case["D"] * float(N) ** 3
    elif kind == "free_energy":
        b, f = one(N, 1)
    else:   # F, h1, gamma in and D0, D1 out; one solve and one response at the least
        b, f = N * N * 5 * 8.0, n * 6.0 * float(N) ** 3
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------------------- 64-bit values


def _zs(e, mu, beta, n):
    """The levels' deviations z_0 .. z_n of the recursion."""
    z = [-beta / 2.0 ** (n + 1) * (e - mu)]
    for _ in range(n):
        z.append(2.0 * z[-1] / (1.0 + z[-1] ** 2))
    return z


def _find_mu(e, beta, nocc, n):
    lo, hi = float(e[0]) - 40.0 / beta, float(e[-1]) + 40.0 / beta
    for _ in range(200):
        mu = 0.5 * (lo + hi)
        if mu in (lo, hi):
            break
        if float((0.5 * (1.0 + _zs(e, mu, beta, n)[-1])).sum()) < nocc:
            lo = mu
        else:
            hi = mu
    return 0.5 * (lo + hi)


def _levels(H0, beta, nocc, n):
    e, V = torch.linalg.eigh(H0)
    mu = _find_mu(e, beta, nocc, n)
    z = _zs(e, mu, beta, n)
    # dP0/dmu per level, and the divided differences of z_n over the steps
    q = 0.25 * beta * (1.0 - z[-1] ** 2) / (1.0 - z[0] ** 2)
    K = torch.full((e.numel(),) * 2, -beta / 2.0 ** (n + 1), dtype=e.dtype, device=e.device)
    for zk in z[:-1]:
        a = 1.0 + zk ** 2
        K = K * (2.0 * (1.0 - zk[:, None] * zk[None, :]) / (a[:, None] * a[None, :]))
    return e, V, mu, z, q, 0.5 * K


def _first_order(V, q, K, H1):
    X = K * (V.T @ H1 @ V)
    mu1 = -float(X.diagonal().sum() / q.sum())
    return X + torch.diag(mu1 * q), mu1


def _exact_solve(H0, H1, beta, nocc, n):
    e, V, mu, z, q, K = _levels(H0, beta, nocc, n)
    P0 = (V * (0.5 * (1.0 + z[-1]))) @ V.T
    P1, pot, alpha = [], [mu], []
    for h in H1:
        X, mu1 = _first_order(V, q, K, h)
        P1.append(V @ X @ V.T)
        pot.append(mu1)
        alpha.append(float(-2.0 * (P1[-1] * h).sum()))
    return P0, torch.stack(P1), np.array(pot), np.array(alpha)


def _second_order(V, e, mu, z, q, K, H1, beta, n):
    """P2 of one direction: orders 1 and 2 of the recursion in the eigenbasis of H0."""
    s2 = beta / 2.0 ** (n + 1)
    X = V.T @ H1 @ V
    _, mu1 = _first_order(V, q, K, H1)
    Z1 = -s2 * (X - mu1 * torch.eye(e.numel(), dtype=e.dtype, device=e.device))
    Z2 = torch.zeros_like(Z1)
    for k in range(n):
        zk, y, a = z[k], z[k + 1], 1.0 + z[k] ** 2
        A1 = zk[:, None] * Z1 + Z1 * zk[None, :]
        A2 = zk[:, None] * Z2 + Z2 * zk[None, :] + Z1 @ Z1
        Y1 = (2.0 * Z1 - A1 * y[None, :]) / a[:, None]
        Z2 = (2.0 * Z2 - A1 @ Y1 - A2 * y[None, :]) / a[:, None]
        Z1 = Y1
    P2 = 0.5 * Z2
    P2 = P2 - torch.diag(float(P2.diagonal().sum() / q.sum()) * q)
    return V @ P2 @ V.T


def exact(case, seed):
    """run()'s outputs from a diagonalisation of H0, in 64 bits. None for the charge loop (its
    fixed point is iterated to a tolerance) and for sizes whose diagonalisation takes too long."""
    kind, n, beta = case["kind"], case["n"], case["beta"]
    if kind == "scc":
        return None
    if kind == "batch":
        g = _gen(seed)
        rs = [_exact_solve(*_cluster(N, g), beta, float(N // 2), n) for N in _cluster_sizes(case)]
        return (*[r[0] for r in rs], *[r[1] for r in rs], np.stack([r[2] for r in rs]),
                np.stack([r[3] for r in rs]))
    if _size(case) > 4500:
        return None
    H0, H1 = _hamiltonian(case, seed)
    nocc = H0.shape[0] / 2.0
    if kind == "solve":
        return _exact_solve(H0, H1, beta, nocc, n)
    e, V, mu, z, q, K = _levels(H0, beta, nocc, n)
    P0 = (V * (0.5 * (1.0 + z[-1]))) @ V.T
    if kind == "adjoint":
        X, _ = _first_order(V, q, K, _sym_normal(H0.shape[0], _gen(seed + 1)))
        return P0, V @ X @ V.T
    if kind == "alpha_grad":
        alpha = [float(-2.0 * (V @ _first_order(V, q, K, h)[0] @ V.T * h).sum()) for h in H1]
        grad = sum(-4.0 * _second_order(V, e, mu, z, q, K, h, beta, n) for h in H1)
        return torch.tensor(alpha, dtype=torch.float64), grad
    # free energy: Tr[P0 H0] - T S with ln(p / (1 - p)) = 2^(n+1) atanh(z_0)
    p = 0.5 * (1.0 + z[-1])
    logit = 2.0 ** (n + 1) * torch.atanh(z[0])
    # -[p ln p + (1 - p) ln(1 - p)] = ln(1 + e^-|logit|) + |logit| (smaller occupation)
    small = torch.sigmoid(-logit.abs())
    entropy = (torch.log1p(torch.exp(-logit.abs())) + logit.abs() * small).sum()
    omega = (p * e).sum() - entropy / beta
    h = e + logit / beta
    dp = -q                                    # dp_i/de_i at fixed mu
    grad = p + h * dp - dp * (h * dp).sum() / dp.sum()
    return omega, (V * grad) @ V.T
